"""jacobi_not_converged counts the patches that hit the sweep cap, not those that share
a warp with one: lists of identical points (converged at once) between lists of
generic ones (not after one sweep)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [9, 16, 24, 32, 40])
def test_only_patches_at_the_cap_are_counted(k):
    from paper_2606_06329_gb300 import _native as N
    from paper_2606_06329_gb300 import api
    rng = np.random.default_rng(k)
    X = np.concatenate([rng.standard_normal((k, 150)), np.zeros((k, 150))])
    n = 2 * k
    generic = np.arange(n) % 5 == 0
    idx = np.where(generic[:, None], np.arange(k)[None, :], np.arange(k, 2 * k)[None, :]).astype(np.int32)
    with api.Context(0) as c:
        c.set_option(N.OPT_JACOBI_MAX_SWEEPS, 1)
        c.mecuco_curvature(torch.from_numpy(X.astype(np.float32)).cuda(), k, idx=torch.from_numpy(idx).cuda(),
                           precision="bf16_mixed")
        torch.cuda.synchronize()
        stats = c.mecuco_get_stats()
        assert c.mecuco_get_last_status() == N.ERR_NOT_CONVERGED
    assert stats["jacobi_not_converged"] == int(generic.sum())
