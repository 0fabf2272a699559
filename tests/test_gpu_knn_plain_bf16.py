"""The plain search on BF16 rows: whole vectors of four, a ragged end, rows and bases on
odd addresses, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from gpu_helpers import knn_mismatches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,ld,first", [(300, 7, 7, 0), (300, 7, 13, 0), (300, 8, 8, 0), (300, 8, 8, 1),
                                          (1025, 65, 68, 0), (1025, 65, 68, 2), (2049, 130, 130, 0), (500, 33, 36, 4)])
@pytest.mark.parametrize("include_self", [False, True])
def test_plain_search_of_bf16_rows(orc, n, m, ld, first, include_self):
    from paper_2606_06329_gb300 import api
    rng = np.random.default_rng(n + m + ld)
    flat = torch.zeros(first + n * ld, dtype=torch.bfloat16, device="cuda")
    X = flat[first:].view(n, ld)[:, :m]
    X.copy_(torch.from_numpy(rng.standard_normal((n, m)).astype(np.float32)).cuda())
    X64 = X.float().cpu().numpy().astype(np.float64)
    k = 17
    with api.Context(0) as c:
        idx = c.mecuco_knn(X, k, include_self=include_self).cpu().numpy()
        assert c.mecuco_get_last_status() == 0
    rows = rng.choice(n, 200, replace=False)
    ref, d = orc.knn(X64, k, rows=rows, include_self=include_self)
    assert knn_mismatches(X64, idx[rows], ref, d, rows=rows) == []
