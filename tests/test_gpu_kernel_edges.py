"""The kernels whose work split depends on the sizes, at the edges of the splits,
against the FP64 oracle: the searches and their re-ranking (lists, chunks of
columns, ties, unaligned rows), the plain FP32 curvature (CTA sizes by k, column
chunks), the third moments from row pairs (all pairs below 128 columns, the pairs
inside two halves of the rows from there) and the gradient's kernels."""
import numpy as np
import pytest
import torch

from gpu_helpers import knn_mismatches, rel_err

pytestmark = pytest.mark.gpu

U_BF16 = 2.0 ** -9


@pytest.fixture(scope="module")
def ctx():
    from paper_2606_06329_gb300 import api
    c = api.Context(0)
    yield c
    c.close()


def _points(n, m, seed, noise=0.3):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, min(m, 8))) @ rng.standard_normal((min(m, 8), m)) / np.sqrt(8)
    return (X + noise * rng.standard_normal((n, m))).astype(np.float32)


# m: one column, below a copy's alignment, one chunk and one more; k: the shortest
# list, the edges of the candidate lists (k + 16 evaluated first, 64 at most kept);
# n: below a tile, a tile's edge, rows left over for a part of a wave
@pytest.mark.parametrize("precision", ["fp32", "bf16_mixed"])
@pytest.mark.parametrize("n,m,k", [(70, 1, 2), (129, 3, 2), (257, 7, 47), (300, 16, 48), (1025, 65, 49),
                                   (2049, 33, 64), (5000, 130, 10), (20011, 40, 63)])
def test_search_edges(ctx, orc, precision, n, m, k):
    X = _points(n, m, n + m)
    idx = ctx.mecuco_knn(torch.from_numpy(X).cuda(), k, precision=precision).cpu().numpy()
    assert ctx.mecuco_get_last_status() == 0
    rows = np.random.default_rng(k).choice(n, min(n, 300), replace=False)
    ref, d = orc.knn(X.astype(np.float64), k, rows=rows)
    assert knn_mismatches(X.astype(np.float64), idx[rows], ref, d, rows=rows) == []


@pytest.mark.parametrize("precision", ["fp32", "bf16_mixed"])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_search_ties_and_padded_rows(ctx, orc, precision, storage):
    # whole numbers (distances exact in both forms), each point four times, rows of
    # an odd stride: distances tie in every list, and the smaller index comes first
    if storage == "bf16" and precision == "fp32":
        pytest.skip("plain search reads FP32 rows here")
    rng = np.random.default_rng(3)
    X = np.repeat(rng.integers(-3, 4, size=(600, 5)), 4, axis=0).astype(np.float32)
    rng.shuffle(X)
    big = torch.zeros((X.shape[0], 13), device="cuda")
    big[:, :5] = torch.from_numpy(X).cuda()
    if storage == "bf16":
        big = big.to(torch.bfloat16)
    k = 21
    idx = ctx.mecuco_knn(big[:, :5], k, precision=precision).cpu().numpy()
    assert ctx.mecuco_get_last_status() == 0
    ref, _ = orc.knn(X.astype(np.float64), k)
    assert np.array_equal(idx, ref)


# k: the edges of the CTA sizes (24, 32, 40; two passes from 49) and of the Gram's
# (40, 60); m: a part of a column chunk, one chunk, one more column, several
@pytest.mark.parametrize("variant", ["literal", "haar"])
@pytest.mark.parametrize("k", [2, 3, 8, 24, 25, 32, 33, 40, 41, 48, 49, 60, 61, 64])
def test_plain_curvature_edges(ctx, orc, k, variant):
    for m in (31, 32, 33, 100):
        X = _points(k + 37, m, 7 * k + m)
        idx, _ = orc.knn(X.astype(np.float64), k)
        got = ctx.mecuco_curvature(torch.from_numpy(X).cuda(), k, idx=torch.from_numpy(idx).cuda(), precision="fp32",
                                   variant=variant, return_s=True, return_lambda=True)
        assert ctx.mecuco_get_last_status() == 0
        ref, terms, lam = orc.curvature(X.astype(np.float64), k, idx, return_terms=True,
                                        variant=orc.HAAR if variant == "haar" else orc.LITERAL)
        t = dict(zip(orc.TERMS, terms.T))
        # the plain form's target, 1e-4, of the terms that are summed (with q = m - p
        # = 1 the null term is a difference of terms of the size of tau)
        q = np.maximum(m - min(k - 1, m), 1)
        scale = np.maximum(np.abs(ref), 0.5 * (t["t_range"] + np.abs(t["t_null"]) + t["tau"]) + 2.0 * t["tau"] / q)
        assert (np.abs(got["kappa"].cpu().numpy() - ref) / scale).max() < 1e-4
        p = min(k - 1, m)
        assert rel_err(got["lambda"].cpu().numpy()[:, :p].sum(1), lam[:, :p].sum(1)).max() < 1e-5


# the boundary of the two tables of pairs, k at the edges of their classes
@pytest.mark.parametrize("variant", ["literal", "haar"])
@pytest.mark.parametrize("m", [127, 128, 129])
def test_third_moment_tables(ctx, orc, m, variant):
    for k in (4, 8, 9, 16, 17, 33, 41, 56, 57, 64):
        X = _points(k + 60, m, k + m, noise=0.6)
        idx, _ = orc.knn(X.astype(np.float64), k)
        got = ctx.mecuco_curvature(torch.from_numpy(X).cuda(), k, idx=torch.from_numpy(idx).cuda(),
                                   precision="bf16_mixed", variant=variant)
        assert ctx.mecuco_get_last_status() == 0
        ref, terms, _ = orc.curvature(X.astype(np.float64), k, idx, return_terms=True,
                                      variant=orc.HAAR if variant == "haar" else orc.LITERAL)
        t = dict(zip(orc.TERMS, terms.T))
        scale = 0.5 * (t["t_range"] + np.abs(t["t_null"]) + t["tau"]) + 2.0 * t["tau"] / (m - k + 1)
        err = np.abs(got.cpu().numpy() - ref) / scale
        # a rounding of Y moves a sum of squares by 8 u of its size at most when all
        # entries move together; they are independent, so the mean over the points
        # stays below that divided by sqrt(k m / 8) (eight standard errors of u / sqrt 3)
        assert err.max() < 8 * U_BF16
        assert err.mean() < 8 * U_BF16 / np.sqrt(k * m / 8)


# k: rows of C not a multiple of 4 or 8, the edges of the CTA sizes (32, 44), block
# columns of more than 32 rows; m: the 128-column chunk and one more column
@pytest.mark.parametrize("variant", ["literal", "haar"])
@pytest.mark.parametrize("k", [2, 5, 7, 12, 31, 32, 33, 41, 44, 45, 57, 64])
def test_gradient_edges(ctx, orc, k, variant):
    from oracle import adjoint as A
    m = 129 if k % 2 else 128
    X = _points(k + 9, m, 11 * k, noise=0.6)
    X64 = X.astype(np.float64)
    idx, _ = orc.knn(X64, k)
    dX = ctx.mecuco_curvature_backward(torch.from_numpy(X).cuda(), k, torch.from_numpy(idx).cuda(),
                                       torch.ones(X.shape[0], device="cuda"), variant=variant)
    assert ctx.mecuco_get_last_status() == 0
    ref = A.grad_adjoint(X64, idx, variant=variant)
    # the gradient's target, 1e-3, on its norm: single coordinates follow the
    # eigenvalue gaps of these patches (test_gpu_grad holds those to their
    # conditioning), a wrong row or block moves the norm by its own size
    err = np.linalg.norm(dX.cpu().numpy() - ref) / np.linalg.norm(ref)
    print(f"gradient k={k} m={m} {variant}: rel err {err:.1e}")
    assert err < 1e-3
