"""Sets of very large and very small numbers, where the products of two entries of the
patch Gram leave FP32's range: every result is the scaled one, exactly (the factor is a
power of two)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


# full-rank patches downwards: the null vectors of the others follow noise of 2^-48 of
# the Gram, which the small scale takes below FP32's range
@pytest.mark.parametrize("m,k,e", [(16, 12, -33), (16, 30, 33), (64, 20, -33), (64, 20, 33), (150, 20, -33),
                                   (150, 20, 33)])
@pytest.mark.parametrize("warp", [-1, 0])
def test_scaled_by_a_power_of_two(m, k, e, warp):
    from paper_2606_06329_gb300 import _native as N
    from paper_2606_06329_gb300 import api
    rng = np.random.default_rng(m + k)
    X = (rng.standard_normal((300, 5)) @ rng.standard_normal((5, m)) + 0.3 * rng.standard_normal((300, m)))
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    c = 2.0 ** e
    with api.Context(0) as ctx:
        ctx.set_option(N.OPT_JACOBI_WARP, warp)
        idx = ctx.mecuco_knn(X, k)
        assert torch.equal(ctx.mecuco_knn(X * c, k), idx)
        for precision in ("fp32", "bf16_mixed"):
            a = ctx.mecuco_curvature(X, k, idx=idx, precision=precision, return_lambda=True, return_U=True)
            b = ctx.mecuco_curvature(X * c, k, idx=idx, precision=precision, return_lambda=True, return_U=True)
            assert ctx.mecuco_get_last_status() == 0
            assert torch.equal(b["U"], a["U"]), precision
            assert torch.equal(b["lambda"], a["lambda"] * c * c), precision
            assert torch.equal(b["kappa"], a["kappa"] * c * c), precision
        if m <= 64:
            a, b = ctx.mecuco_curvature_exact(X, k, idx=idx), ctx.mecuco_curvature_exact(X * c, k, idx=idx)
            assert torch.equal(b, a * c * c)
