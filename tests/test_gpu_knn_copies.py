"""Clusters off the origin that hold many copies of one point.  The search gives the
copies one common error, and where that happens to be low they are the nearest of
the lists for every other point of the cluster: an error estimated from the nearest
candidates alone is then that of a single point.  Every list is held to the FP64
distances."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2606_06329_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def _data(m, copies, seed):
    """40 clusters of 38 points and `copies` more of the first; columns around 1, distances
    of about 1e-7 of the squared norm, 1% apart."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rows = []
    for c in range(40):
        centre = 1.0 + 0.5 * torch.randn(m, generator=g, device="cuda", dtype=torch.float64)
        p = centre + 2.0 ** -12 * torch.randn(38, m, generator=g, device="cuda", dtype=torch.float64)
        rows += [p, p[:1].expand(copies, m)]
    X = torch.cat(rows)
    return X[torch.randperm(len(X), generator=g, device="cuda")].float()


@pytest.mark.parametrize("precision", ["fp32", "bf16_mixed"])
@pytest.mark.parametrize("m", [1024, 4096, 20000])
def test_copies_off_the_origin(ctx, precision, m):
    bad = {}
    for seed in (1, 2, 3):
        X = _data(m, 22, seed)
        x = X.double()
        x = x - 1.0
        sq = x.square().sum(1)
        d = sq[:, None] + sq[None, :] - 2.0 * x @ x.T
        for a in range(0, len(X), 100):  # near pairs by differences
            b = min(a + 100, len(X))
            near = d[a:b].topk(64, largest=False).indices
            e = (x[near] - x[a:b, None]).square().sum(2) if m <= 4096 else torch.stack(
                [(x[near[i]] - x[a + i]).square().sum(1) for i in range(b - a)])
            d[a:b].scatter_(1, near, e)
        d.fill_diagonal_(float("inf"))
        for k in (2, 4):
            idx = ctx.mecuco_knn(X, k, precision=precision)
            assert ctx.mecuco_get_last_status() == 0
            unc = ctx.mecuco_get_stats()["knn_uncertified"]
            best = d.topk(k, largest=False).values
            got = d.gather(1, idx.long()).sort(1).values
            w = int(((got - best).abs() > 1e-6 * best.abs() + 1e-20).any(1).sum())
            print(f"{precision} m={m} seed={seed} k={k}: {w} wrong, {unc} uncertified of {len(X)}")
            if w:
                bad[(seed, k)] = w
    assert not bad
