"""Points much closer to each other than the search resolves (rows of norm 64, distances
of 2^-15): the exact re-rank must order them all the same.  Every point has a twin whose
distances differ from its own by about 2^-29 relative, far above the re-rank's
rounding (2^-42) and far below FP32's."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _twins(m, seed):
    rng = np.random.default_rng(seed)
    rows = []
    for c in range(3):
        centre = 1.0 + 0.5 * rng.standard_normal(m)
        centre[0] = 2.0 ** -12
        y = centre + 2.0 ** -14 * rng.standard_normal((30, m))
        y[:, 0] = 2.0 ** -12 + 2.0 ** -16 * rng.standard_normal(30)
        y = y.astype(np.float32)
        z = y.copy()
        z[:, 0] += 64 * np.spacing(y[:, 0])
        rows += [y, z]
    X = np.concatenate(rows)
    return X[rng.permutation(len(X))]


@pytest.mark.parametrize("precision", ["fp32", "bf16_mixed"])
@pytest.mark.parametrize("pad", [0, 1])  # rows on 16-byte boundaries, and not
def test_order_far_below_the_search_distance(precision, pad):
    from paper_2606_06329_gb300 import api
    m, k = 4096, 20
    X = _twins(m, 3)
    X64 = X.astype(np.float64)
    d = np.stack([np.square(X64 - X64[q]).sum(1) for q in range(len(X))])
    np.fill_diagonal(d, np.inf)
    big = torch.zeros((len(X), m + pad), device="cuda")
    big[:, :m] = torch.from_numpy(X).cuda()
    with api.Context(0) as ctx:
        idx, dist = ctx.mecuco_knn(big[:, :m], k, precision=precision, return_dist=True)
        assert ctx.mecuco_get_last_status() == 0
    idx, dist = idx.cpu().numpy(), dist.cpu().numpy().astype(np.float64)
    got = np.take_along_axis(d, idx, 1)
    best = np.sort(d, 1)[:, :k]
    worst = np.abs(got / best - 1.0).max()
    print(f"{precision} pad={pad}: largest relative error of a position {worst:.2e}, "
          f"of a distance {np.abs(dist / got - 1.0).max():.2e}")
    assert worst < 2.0 ** -38
    assert np.abs(dist / got - 1.0).max() < 2.0 ** -23.9  # rounded once
