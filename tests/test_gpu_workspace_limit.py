"""Searches under MECUCO_OPT_WORKSPACE_LIMIT: where the fastest split of the candidates
needs more lists than the limit allows, the call takes fewer, down to one list set per
row, and gives the same neighbours."""
import pytest
import torch

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _x(n, m, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, m, generator=g, device="cuda").to(dtype)


# the limit: above the smallest workspace, below that of the split taken without one
@pytest.mark.parametrize("n,m,dtype,precision,k,limit", [
    (10000, 784, torch.float32, "fp32", 32, 21 * MB),
    (10000, 784, torch.float32, "fp32", 32, 6 * MB),
    (15000, 512, torch.bfloat16, "bf16_mixed", 40, 32 * MB),
    (15000, 512, torch.bfloat16, "bf16_mixed", 40, 17 * MB),
    (3000, 64, torch.float32, "bf16_mixed", 10, 8 * MB),
])
def test_fewer_splits_under_a_limit(n, m, dtype, precision, k, limit):
    from paper_2606_06329_gb300 import _native as N
    from paper_2606_06329_gb300 import api
    X = _x(n, m, dtype, n + m)
    with api.Context(0) as c:
        ref = c.mecuco_knn(X, k, precision=precision)
    with api.Context(0) as c:
        c.set_option(N.OPT_WORKSPACE_LIMIT, limit)
        idx = c.mecuco_knn(X, k, precision=precision)
        assert c.mecuco_get_last_status() == 0
        assert torch.equal(idx, ref)
        part = c.mecuco_knn_range(X, k, 100, n - 55, precision=precision)
        assert torch.equal(part, ref[100:n - 55])
        c.set_option(N.OPT_WORKSPACE_LIMIT, 0)
        again = c.mecuco_knn(X, k, precision=precision)  # the option off: the fastest split again
        assert torch.equal(again, ref)
        assert c.mecuco_get_last_status() == 0


def test_whole_calls_under_a_limit():
    from paper_2606_06329_gb300 import _native as N
    from paper_2606_06329_gb300 import api
    X = _x(6000, 40, torch.float32, 5)
    with api.Context(0) as c:
        ref = c.mecuco_curvature(X, 20)
        host = c.mecuco_curvature_host(X.cpu(), 20)
        lanes = [v.clone() for v in c.mecuco_curvature_batched([X, X[:2500]], [20, 12], precision="fp32")]
    with api.Context(0) as c:
        # lists of one split: 6,000 x 64 entries of 8 bytes; the estimator's buffers: 40 MB
        c.set_option(N.OPT_WORKSPACE_LIMIT, 45 * MB)
        assert torch.equal(c.mecuco_curvature(X, 20), ref)
        assert torch.equal(c.mecuco_curvature_host(X.cpu(), 20), host)
        c.set_option(N.OPT_WORKSPACE_LIMIT, 70 * MB)
        got = c.mecuco_curvature_batched([X, X[:2500]], [20, 12], precision="fp32")
        assert all(torch.equal(a, b) for a, b in zip(got, lanes))
        assert c.mecuco_get_last_status() == 0
