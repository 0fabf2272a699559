"""Searches whose distances are small beside the rows' norms: the case in which the
search's accumulation error is of the size of the gaps between neighbours, so that a
list is right only if the certificate notices it (csrc/knn_simt.cu).  Every list is
held to the FP64 distances; the number of rows that went to the exact scan is
printed."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2606_06329_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def _clusters(n, m, noise, seed, shuffled):
    """Four clusters off the origin, the energy of the columns falling as
    1 / sqrt(1 + a / 4) (principal components, spectra, wavelet coefficients)."""
    g = torch.Generator().manual_seed(seed)
    scale = (1.0 + torch.arange(m) / 4.0).rsqrt()
    centres = torch.randn(4, m, generator=g) * scale
    rms = centres.square().mean(1).sqrt()
    of = torch.arange(4).repeat_interleave(n // 4)
    if shuffled:
        of = of[torch.randperm(len(of), generator=g)]
    return centres[of] + noise * rms[of][:, None] * torch.randn(len(of), m, generator=g)


def _wrong(X, idx, k, tie_rel=1e-6):
    """Rows whose neighbours' FP64 distances are not the k smallest."""
    x = X.double()
    x = x - x.mean(0)  # smaller norms; FP64 leaves 1e-13 of them
    sq = x.square().sum(1)
    d = sq[:, None] + sq[None, :] - 2.0 * x @ x.T
    d.fill_diagonal_(float("inf"))
    best = d.topk(k, largest=False).values
    got = d.gather(1, idx.long()).sort(1).values
    scale = best.abs().clamp_min(1e-300)
    return int(((got - best).abs() / scale > tie_rel).any(1).sum())


@pytest.mark.parametrize("storage,m", [("bf16", 1024), ("bf16", 4096), ("f32", 784)])
@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("splits", [0, 1])
def test_clusters_off_the_origin(ctx, storage, m, shuffled, splits):
    from paper_2606_06329_gb300 import _native as N
    bad = {}
    ctx.set_option(N.OPT_KNN_SPLITS, splits)
    try:
        for noise in (0.008, 0.0125, 0.02):
            X = _clusters(2048, m, noise, int(1e5 * noise) + m, shuffled).cuda()
            if storage == "bf16":
                X = X.to(torch.bfloat16)
            for k in (2, 5, 10):
                idx = ctx.mecuco_knn(X, k, precision="bf16_mixed")
                assert ctx.mecuco_get_last_status() == 0
                unc = ctx.mecuco_get_stats()["knn_uncertified"]
                w = _wrong(X, idx, k)
                print(f"{storage} m={m} noise={noise} k={k} shuffled={shuffled} splits={splits}: "
                      f"{w} wrong, {unc} uncertified of {X.shape[0]}")
                if w:
                    bad[(noise, k)] = w
    finally:
        ctx.set_option(N.OPT_KNN_SPLITS, 0)
    assert not bad


@pytest.mark.parametrize("precision,storage", [("bf16_mixed", "bf16"), ("bf16_mixed", "f32"), ("fp32", "f32"),
                                               ("fp32", "bf16")])
@pytest.mark.parametrize("m", [64, 1000, 4096])
def test_many_near_equal_distances(ctx, precision, storage, m):
    # independent columns: all distances lie within a few times m^-1/2 of each
    # other; the further off the origin, the more of their gaps the search's error covers
    bad = {}
    for offset in (1.0, 4.0, 16.0, 64.0):
        g = torch.Generator().manual_seed(m + int(offset))
        X = (offset * (1.0 + 0.1 * torch.randn(m, generator=g)) + torch.randn(3000, m, generator=g)).cuda()
        if storage == "bf16":
            X = X.to(torch.bfloat16)
        for k in (2, 20, 64):
            idx = ctx.mecuco_knn(X, k, precision=precision)
            assert ctx.mecuco_get_last_status() == 0
            unc = ctx.mecuco_get_stats()["knn_uncertified"]
            w = _wrong(X, idx, k)
            print(f"{precision} {storage} m={m} offset={offset} k={k}: {w} wrong, {unc} uncertified of 3000")
            if w:
                bad[(offset, k)] = w
    assert not bad
