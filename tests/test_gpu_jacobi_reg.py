"""The register-resident one-sided eigensolve (jacobi_reg.cu, the default sweeps
wherever a refinement step follows) at the edges of its column classes
(R = 16, 24, ..., 64), for full-rank, rank-deficient and all-equal patches."""
import numpy as np
import pytest
import torch

from gpu_helpers import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2606_06329_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def _check(ctx, orc, X, k, deficient):
    N = X.shape[0]
    Xd = torch.from_numpy(X).cuda()
    idx = ctx.mecuco_knn(Xd, k)
    o = ctx.mecuco_curvature(Xd, k, idx=idx, precision="bf16_mixed", return_U=True, return_s=True)
    kap = ctx.mecuco_curvature(Xd, k, idx=idx, precision="fp32")
    torch.cuda.synchronize()
    assert ctx.mecuco_get_last_status() == 0
    U = o["U"].double()
    eye = torch.eye(k, device="cuda", dtype=torch.float64)
    # the refinement squares the sweeps' error (columns orthogonal to 2^-10 at
    # worst before the last sweep's own squaring, and to 2^-24 k after it)
    assert float((U.transpose(1, 2) @ U - eye).abs().max()) < 5e-5
    s = o["s"].double()
    assert bool((s[:, 1:] <= s[:, :-1]).all())
    if not deficient:
        ref = orc.curvature(X.astype(np.float64), k, idx.cpu().numpy())
        assert rel_err(kap.cpu().numpy(), ref).max() < 1e-4  # the plain form's target


@pytest.mark.parametrize("k", [2, 3, 15, 16, 17, 24, 25, 32, 33, 40, 41, 48, 49, 56, 57, 63, 64])
@pytest.mark.parametrize("m", [128, 193])
def test_column_classes(ctx, orc, k, m):
    rng = np.random.default_rng(100 * k + m)
    # odd number of points: a last warp with fewer patches than it can hold
    X = (rng.standard_normal((151, 6)) @ rng.standard_normal((6, m)) / 3 + 0.05 * rng.standard_normal((151, m)))
    _check(ctx, orc, X.astype(np.float32), k, False)


@pytest.mark.parametrize("k", [16, 31, 64])
def test_rank_deficient(ctx, orc, k):
    rng = np.random.default_rng(k)
    X = (rng.standard_normal((131, 5)) @ rng.standard_normal((5, 140))).astype(np.float32)  # rank 5 and rounding
    _check(ctx, orc, X, k, True)
    # copies of a few points: zero and rank-one patches
    Y = np.repeat(rng.standard_normal((2, 130)).astype(np.float32), 70, axis=0)
    _check(ctx, orc, Y, k, True)


def test_scale(ctx):
    # the solve scales by a power of two: K(c X) = c^2 K(X) holds exactly for c = 2^e
    rng = np.random.default_rng(9)
    X = torch.from_numpy(rng.standard_normal((200, 133)).astype(np.float32)).cuda()
    idx = ctx.mecuco_knn(X, 20)
    a = ctx.mecuco_curvature(X, 20, idx=idx, precision="bf16_mixed")
    for e in (-20, 20):
        b = ctx.mecuco_curvature(X * 2.0 ** e, 20, idx=idx, precision="bf16_mixed")
        assert torch.equal(b, a * 2.0 ** (2 * e))
