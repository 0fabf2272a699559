"""A host-side model of the estimated part of the kNN certificate
(csrc/knn_simt.cu, knn_rerank_kernel) on searches whose accumulation error is as
large as the gaps between neighbours.

The search's distances d~ carry the rounding of its FP32 accumulation.  Nothing
useful bounds that a priori, so the certificate estimates it per row from candidates
whose exact distances it has: the largest overestimate + three times the spread of
d~ - d, plus 2^-21 of the norms; FP32 rows add a bound on what their BF16 terms leave
out.  The estimate holds as far as the evaluated candidates show what errors the
others have, so besides the nearest a fixed sample of the lists is evaluated.  The model restates the search (tiles of
256 candidates, two lists of 64 a row by column half, an accumulator that adds exact
sums of 16 products and truncates to FP32) and the certificate, and counts the rows
that come out certified with a wrong list.  The kernel's form must leave none.  Two
others are caught: the K blocks of every second tile in descending order (an error by
the parity of the tile, which the nearest candidates of one parity do not show), and
the nearest candidates without the sample (copies of one point show one error)."""
import numpy as np
import pytest

from paper_2606_06329_gb300 import synth

RR_EXTRA, RR_SAMPLE = 16, 16
TILE, CAP = 256, 64


def _bf16(x):
    return synth.bf16_bits_to_f32(synth.f32_to_bf16_bits(np.asarray(x, np.float32)))


def _terms(X):
    """h and l of the split x = h + l + r."""
    h = _bf16(X)
    return h, _bf16(X - h)


def _apriori(X):
    """Per row, the bound on what the split's products leave out of a dot product."""
    x64 = X.astype(np.float64)
    h, l = (v.astype(np.float64) for v in _terms(X))
    norm = [np.sqrt(np.square(v).sum(1)) for v in (x64, l, x64 - h - l)]
    (xn, t1, t2), (ym, m1, m2) = norm, [v.max() for v in norm]
    return 2.0 * (t1 * m1 + (xn + t2) * m2 + t2 * (ym + m2) + t2 * m2) + (xn ** 2 + ym ** 2) * 2.0 ** -21


def _trunc32(v):
    """FP64 values truncated to FP32 precision."""
    f = v.astype(np.float32)
    over = np.abs(f.astype(np.float64)) > np.abs(v)
    return np.where(over, np.nextafter(f, np.float32(0.0)), f).astype(np.float64)


def _search_tc(X, rows, alternate=False, split=False):
    """d~ of the tensor-core search: sums of 16 products, truncated to FP32 as they are
    added; with `alternate` the blocks of 32 columns descend on odd tiles; with `split`
    FP32 rows as the three-term operands [h | h | l] and [h | l | h]."""
    x64 = X.astype(np.float64)
    a64 = b64 = x64
    if split:
        h, l = (v.astype(np.float64) for v in _terms(X))
        a64, b64 = np.concatenate([h, h, l], 1), np.concatenate([h, l, h], 1)
    n, m = a64.shape
    dot = np.empty((len(rows), n))
    for t in range(0, n, TILE):
        blocks = np.arange(0, m, 32)
        if alternate and (t // TILE) & 1:
            blocks = blocks[::-1]
        acc = np.zeros((len(rows), min(TILE, n - t)))
        for b in blocks:
            for a in (b, b + 16):
                acc = _trunc32(acc + a64[rows, a:a + 16] @ b64[t:t + TILE, a:a + 16].T)
        dot[:, t:t + TILE] = acc
    norms = np.square(x64).sum(1).astype(np.float32)
    s = (norms[rows][:, None] + norms[None, :]).astype(np.float32)  # FP32 sum, then one FMA
    return (s.astype(np.float64) - 2.0 * dot).astype(np.float32)


def _lists(dt, q, halves):
    """The listed candidates of a row and the smallest maximum of the full lists."""
    n = len(dt)
    cols = np.arange(n)
    listed, thr = [], np.inf
    for h in range(halves):
        c = cols[(cols % TILE) // (TILE // halves) == h]
        c = c[c != q]
        keep = np.sort(c[np.argsort(dt[c], kind="stable")[:CAP]])
        if len(c) >= CAP:
            thr = min(thr, float(dt[keep].max()))
        listed.append(keep)
    return np.concatenate(listed), thr


def _certified_list(X64, norms, dt, q, k, halves, sample, apriori):
    """The re-rank's list of row q and whether it is certified."""
    cand, thr = _lists(dt, q, halves)
    exact = np.square(X64[cand] - X64[q]).sum(1)
    err = dt[cand].astype(np.float64) - exact
    order = np.argsort(dt[cand], kind="stable")
    done = np.zeros(len(cand), bool)
    done[order[:k + RR_EXTRA]] = True
    if sample:
        done[::-(-len(cand) // RR_SAMPLE)] = True  # each list is in the order of its candidates here
        done[dt[cand] == dt[cand].max()] = True
    while True:
        e = err[done]
        ev = cand[done]
        best = ev[np.lexsort((ev, exact[done]))[:k]]
        theta = np.sort(exact[done])[k - 1]
        nmax = max(norms[ev].max(), (np.sqrt(norms[q]) + np.sqrt(theta)) ** 2)
        e_hi = max(max(e.max(), 0.0) + 3.0 * (e.max() - e.min()) + (norms[q] + nmax) * 2.0 ** -21, apriori)
        more = ~done & (dt[cand] <= theta + e_hi)
        if not more.any():
            break
        done |= more
    return best, thr - e_hi > theta


def _clusters(n, m, noise, seed):
    rng = np.random.default_rng(seed)
    scale = 1.0 / np.sqrt(1.0 + np.arange(m) / 4.0)
    centres = rng.standard_normal((4, m)) * scale
    rms = np.sqrt(np.square(centres).mean(1))
    of = np.repeat(np.arange(4), n // 4)
    X = centres[of] + noise * rms[of][:, None] * rng.standard_normal((n, m))
    return _bf16(X)


def _count(X, rows, dt, k, halves, sample=True, apriori=None):
    """(certified and wrong, uncertified) of the rows."""
    X64 = X.astype(np.float64)
    norms = np.square(X64).sum(1)
    wrong = unc = 0
    for i, q in enumerate(rows):
        got, ok = _certified_list(X64, norms, dt[i], q, k, halves, sample,
                                  -np.inf if apriori is None else apriori[q])
        d = np.square(X64 - X64[q]).sum(1)
        d[q] = np.inf
        if not ok:
            unc += 1
        elif np.abs(np.sort(d[got]) - np.sort(d)[:k]).max() > 1e-6 * np.sort(d)[k - 1]:
            wrong += 1
    return wrong, unc


@pytest.mark.parametrize("m,noise", [(4096, 0.0125)])
def test_one_order_of_the_columns_for_every_tile(m, noise):
    X = _clusters(2048, m, noise, m)  # a cluster spans two tiles
    rows = np.random.default_rng(1).choice(len(X), 24, replace=False)
    kernel, planted = _search_tc(X, rows, False), _search_tc(X, rows, True)
    caught = 0
    for k in (2, 5, 10):
        wrong, unc = _count(X, rows, kernel, k, 2)
        pw, pu = _count(X, rows, planted, k, 2, False)
        print(f"m={m} noise={noise} k={k}: one order {wrong} wrong, {unc} uncertified; "
              f"alternating {pw} wrong, {pu} uncertified of {len(rows)}")
        assert wrong == 0
        caught += pw
    assert caught > len(rows)


def test_a_sample_beside_the_nearest():
    # clusters of 8 points and 30 more copies of the first, distances of 1e-7 of the norms
    rng = np.random.default_rng(5)
    parts = []
    for _ in range(24):
        p = 1.0 + 0.5 * rng.standard_normal(1024) + 2.0 ** -12 * rng.standard_normal((8, 1024))
        parts += [p, np.repeat(p[:1], 30, axis=0)]
    X = np.concatenate(parts)
    single = np.tile(np.arange(38) % 38, 24)
    mix = rng.permutation(len(X))
    X, single = X[mix].astype(np.float32), single[mix]
    rows = np.flatnonzero((single > 0) & (single < 8))
    dt, apriori = _search_tc(X, rows, split=True), _apriori(X)
    wrong, unc = _count(X, rows, dt, 2, 2, True, apriori)
    nw, nu = _count(X, rows, dt, 2, 2, False, apriori)
    print(f"with the sample {wrong} wrong, {unc} uncertified; the nearest alone {nw} wrong, {nu} uncertified "
          f"of {len(rows)}")
    assert wrong == 0
    assert nw > 0
