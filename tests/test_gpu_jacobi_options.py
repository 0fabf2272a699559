"""MECUCO_OPT_JACOBI_WARP selects the sweeps it names on every path: 2 is the fused form
with two warps per patch, which applies the same rotations as that with one or four;
-1 (the default) the register-resident one-sided form where only refined eigenpairs
are used."""
import numpy as np
import pytest
import torch

from gpu_helpers import rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [12, 33])
def test_forms_by_option(orc, k):
    from paper_2606_06329_gb300 import _native as N
    from paper_2606_06329_gb300 import api
    rng = np.random.default_rng(k)
    X = (rng.standard_normal((600, 7)) @ rng.standard_normal((7, 160)) + 0.2 * rng.standard_normal((600, 160)))
    X = X.astype(np.float32)
    Xd = torch.from_numpy(X).cuda()
    rot, kap, plain = {}, {}, {}
    with api.Context(0) as c:
        idx = c.mecuco_knn(Xd, k)
        for form in ("unset", -1, 1, 2, 4, -1):
            if form != "unset":
                c.set_option(N.OPT_JACOBI_WARP, form)
            kap[form] = c.mecuco_curvature(Xd, k, idx=idx, precision="bf16_mixed")
            rot[form] = c.mecuco_get_stats()["jacobi_rotations"]
            plain[form] = c.mecuco_curvature(Xd, k, idx=idx, precision="fp32")
            assert c.mecuco_get_last_status() == 0
        for bad in (-2, 3, 5):
            with pytest.raises(N.MecucoError):
                c.set_option(N.OPT_JACOBI_WARP, bad)
    print(f"k={k}: rotations {rot}")
    assert abs(rot[2] - rot[1]) < 0.01 * rot[1] and abs(rot[2] - rot[4]) < 0.01 * rot[4]
    assert rot["unset"] == rot[-1] and torch.equal(kap["unset"], kap[-1]) and torch.equal(plain["unset"], plain[-1])
    assert abs(rot[-1] - rot[2]) > 0.01 * rot[2]
    ref = orc.curvature(X.astype(np.float64), k, idx.cpu().numpy())
    for form in plain:
        assert rel_err(plain[form].cpu().numpy(), ref).max() < 1e-4
        assert rel_err(kap[form].cpu().numpy(), kap[2].cpu().numpy()).max() < 5e-4
