"""Rows with more equal distances than the re-rank holds at a time (128): 225 corners
of a simplex around every point, four such sets.  The lists hold them all and points
beyond, so every row is certified and none needs the exact scan; the neighbours are
the ten smallest indices of the point's set."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "bf16_mixed"])
@pytest.mark.parametrize("include_self", [False, True])
def test_more_ties_than_the_rerank_holds(precision, include_self):
    from paper_2606_06329_gb300 import _native as N
    from paper_2606_06329_gb300 import api
    rng = np.random.default_rng(4)
    of = rng.permutation(np.repeat(np.arange(4), 225))
    X = np.zeros((900, 229), np.float32)
    nth = np.zeros(4, int)
    for i, c in enumerate(of):
        X[i, nth[c]] = 1.0
        X[i, 225 + c] = 4.0
        nth[c] += 1
    with api.Context(0) as ctx:
        ctx.set_option(N.OPT_KNN_SPLITS, 8)  # 113 points to a list: a quarter of them tie
        idx = ctx.mecuco_knn(torch.from_numpy(X).cuda(), 10, precision=precision, include_self=include_self)
        assert ctx.mecuco_get_last_status() == 0
        assert ctx.mecuco_get_stats()["knn_uncertified"] == 0
    for i in range(900):
        same = np.flatnonzero(of == of[i])
        same = same[same != i]
        ref = np.concatenate([[i], same])[:10] if include_self else same[:10]
        assert np.array_equal(idx[i].cpu().numpy(), ref)
