"""Rows that are not finite: every output of a patch that holds one says so, and none
returns what an earlier call left in the workspace; the other patches are untouched.
Below 128 columns the two-sided eigensolve, from there the register-resident one."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 3e38])
@pytest.mark.parametrize("precision", ["fp32", "bf16_mixed"])
@pytest.mark.parametrize("m,k", [(40, 12), (200, 12), (200, 33), (130, 64)])
def test_patches_with_a_non_finite_row(m, k, precision, value):
    from paper_2606_06329_gb300 import _native as N
    from paper_2606_06329_gb300 import api
    rng = np.random.default_rng(m + k)
    n = 300
    X = rng.standard_normal((n, 6)) @ rng.standard_normal((6, m)) + 0.3 * rng.standard_normal((n, m))
    X = torch.from_numpy(X.astype(np.float32)).cuda()
    idx = torch.from_numpy(np.stack([rng.choice(n, k, replace=False) for _ in range(n)]).astype(np.int32)).cuda()
    bad = X.clone()
    bad[17, 3] = value
    bad[17, m - 1] = -value  # the difference of two large values overflows as well
    hit = (idx == 17).any(1)
    assert 0 < int(hit.sum()) < n
    with api.Context(0) as c:
        for form in (2, 0):  # the default and the CTA form of the sweeps
            if form == 0:
                c.set_option(N.OPT_JACOBI_WARP, 0)
            kw = dict(idx=idx, precision=precision, return_lambda=True, return_s=True, return_U=True)
            clean = {a: b.clone() for a, b in c.mecuco_curvature(X, k, **kw).items()}
            got = c.mecuco_curvature(bad, k, **kw)
            for name in ("kappa", "lambda", "s", "U"):
                assert bool(torch.isfinite(clean[name]).all())
                rest = got[name][~hit], clean[name][~hit]
                assert torch.equal(*rest), name
                g = got[name][hit].reshape(int(hit.sum()), -1)
                if value != value:
                    assert not bool(torch.isfinite(g).any()), name
                elif name == "kappa":
                    assert not bool(torch.isfinite(g).any())
                old = clean[name][hit].reshape(g.shape)
                # nothing of an earlier call: a value that is finite is not its
                same = torch.isfinite(g) & (g == old) & (g != 0)
                assert not bool(same.any()), name
