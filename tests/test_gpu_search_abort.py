"""Waits of the tensor-core search that run out at different points of its work (the
first tile, mid-sweep, a later work item), by limits from one clock cycle up: the
launch returns with MECUCO_ERR_TIMEOUT or completes, and the next call gives the
clean run's lists, with one and with several candidate splits per query block."""
import numpy as np
import pytest
import torch

from paper_2606_06329_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("splits", [0, 1, 4])
def test_short_waits_at_any_point(splits):
    from paper_2606_06329_gb300 import _native as N
    from paper_2606_06329_gb300 import api
    n, k = 4000, 20
    bits = synth.curved_patches(n=n, m=512, n_patches=2, seed=77)
    X = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
    with api.Context(0) as c:
        c.set_option(N.OPT_KNN_SPLITS, splits)
        ref = c.mecuco_knn(X, k, precision="bf16_mixed")
        assert c.mecuco_get_last_status() == N.OK
        for limit in (1, 50, 500, 2000, 8000, 30000, 100000):
            c.set_option(N.OPT_WAIT_LIMIT, limit)
            c.mecuco_knn(X, k, precision="bf16_mixed")
            torch.cuda.synchronize()
            assert c.mecuco_get_last_status() in (N.OK, N.ERR_TIMEOUT)
            c.set_option(N.OPT_WAIT_LIMIT, 0)
            again = c.mecuco_knn(X, k, precision="bf16_mixed")
            assert c.mecuco_get_last_status() == N.OK
            assert torch.equal(ref, again)
