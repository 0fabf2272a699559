"""Workloads of the library's main path, for timing and for comparing outputs.

Every case is one call sequence of a user's program on device-resident inputs
through the Python binding (``api.context``, ``autograd.curvature``): neighbour
search, Fast-mode curvature on given lists, the two together on a row range of
a large set, many datasets in one call, the Exact mode, the gradient and the
tangent bases.  Shapes are those of the benchmark (1,000,000 x 4096, k = 64;
70,000 x 784, k = 50; the MLP image batches), of the package's usage example
(100,000 x 512, k = 32), of the decoder and sphere workloads, and odd sizes
between them.  Inputs follow the recipes of ``synth`` but are drawn on the GPU.

``listed()`` gives the named cases, ``draw(rng)`` further ones of the same
ranges, ``prepare``/``run`` one state and one pass, ``work`` the bytes and
operations a pass cannot do without, ``exact`` the same outputs in FP64.
"""
import math

import numpy as np
import torch

from paper_2606_06329_gb300 import api, autograd

DEV = "cuda:0"


def listed():
    return [
        # The smallest calls: a few thousand low-dimensional points, search and
        # curvature as two calls; latency and launches count.
        {"name": "knn_fp32_sphere_2k", "kind": "knn", "data": "sphere", "n": 2000, "m": 32, "k": 10, "dtype": "f32",
         "prec": "fp32"},
        {"name": "curv_fp32_sphere_2k", "kind": "curvature", "data": "sphere", "n": 2000, "m": 32, "k": 10,
         "dtype": "f32", "prec": "fp32", "variant": "literal"},
        # The automatic mode below 50 columns (Theorem 1), search included.
        {"name": "exact_mode_20k", "kind": "exact", "data": "mlp", "n": 20000, "m": 24, "k": 32, "dtype": "f32",
         "prec": "fp32"},
        # Plain FP32 search of an ordinary set.
        {"name": "knn_fp32_50k_256", "kind": "knn", "data": "decoder", "n": 50000, "m": 256, "k": 32, "dtype": "f32",
         "prec": "fp32"},
        # The search of the usage example: BF16 rows on the tensor cores.
        {"name": "knn_bf16_100k_512", "kind": "knn", "data": "curved", "n": 100000, "m": 512, "k": 32,
         "dtype": "bf16", "prec": "bf16_mixed"},
        # FP32 rows searched on the tensor cores (image-like rows, 80% zeros).
        {"name": "knn_f32rows_70k_784", "kind": "knn", "data": "sparse", "n": 70000, "m": 784, "k": 50,
         "dtype": "f32", "prec": "bf16_mixed"},
        # Curvature on given lists, plain FP32 form (decoder workload).
        {"name": "curv_fp32_20k_256", "kind": "curvature", "data": "decoder", "n": 20000, "m": 256, "k": 32,
         "dtype": "f32", "prec": "fp32", "variant": "literal"},
        # The same in the BF16-mixed form on FP32 rows at odd sizes, Haar variant.
        {"name": "curv_mixed_odd_30k_301", "kind": "curvature", "data": "mlp", "n": 29989, "m": 301, "k": 37,
         "dtype": "f32", "prec": "bf16_mixed", "variant": "haar"},
        # Curvature on given lists at the benchmark's width and neighbour count.
        {"name": "curv_bf16_6k_4096", "kind": "curvature", "data": "curved", "n": 6144, "m": 4096, "k": 64,
         "dtype": "bf16", "prec": "bf16_mixed", "variant": "literal"},
        # The gradient (forward and backward through autograd).
        {"name": "grad_fp32_8k_256", "kind": "grad", "data": "mlp", "n": 8000, "m": 256, "k": 32, "dtype": "f32",
         "variant": "literal"},
        # Many uneven datasets in one call.
        {"name": "batched_mlp_12", "kind": "batched", "sets": 12, "shape_seed": 5, "nmax": 20000, "prec": "bf16_mixed"},
        # The benchmark workload: one rank's sixteenth of its query rows against
        # every point, search and curvature (the largest case).
        {"name": "whole_bf16_1m_4096_shard", "kind": "whole", "data": "curved", "n": 1000000, "m": 4096, "k": 64,
         "dtype": "bf16", "rows": 62500, "prec": "bf16_mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["knn", "knn", "curvature", "curvature", "exact", "grad", "batched", "whole"])
    if kind == "knn":
        prec = rng.choice(["fp32", "bf16_mixed"])
        dtype = rng.choice(["f32", "bf16"]) if prec == "bf16_mixed" else "f32"
        n = _log_int(rng, 1000, 50000 if prec == "fp32" else 100000)
        m = _log_int(rng, 16, 512 if prec == "fp32" else 1024)
        data = "curved" if dtype == "bf16" else rng.choice(["mlp", "sparse"])
        return {"kind": kind, "data": data, "n": n, "m": m, "k": rng.randint(5, 64), "dtype": dtype, "prec": prec}
    if kind == "curvature":
        prec = rng.choice(["fp32", "bf16_mixed"])
        dtype = rng.choice(["f32", "bf16"]) if prec == "bf16_mixed" else "f32"
        m = _log_int(rng, 32, 512 if prec == "fp32" else 4096)
        k = rng.randint(5, 64)
        n = _log_int(rng, 1000, max(2000, min(30000, int(3e11 / (m * k ** 3)))))
        return {"kind": kind, "data": "curved" if dtype == "bf16" else "mlp", "n": n, "m": m, "k": k, "dtype": dtype,
                "prec": prec, "variant": rng.choice(["literal", "haar"])}
    if kind == "exact":
        m = rng.randint(6, 48)
        return {"kind": kind, "data": "mlp", "n": _log_int(rng, 1000, 20000), "m": m, "k": rng.randint(m + 4, 64),
                "dtype": "f32", "prec": "fp32"}
    if kind == "grad":
        return {"kind": kind, "data": "mlp", "n": _log_int(rng, 500, 4000), "m": _log_int(rng, 64, 300),
                "k": rng.randint(6, 40), "dtype": "f32", "variant": rng.choice(["literal", "haar"])}
    if kind == "batched":
        return {"kind": kind, "sets": rng.randint(2, 10), "shape_seed": rng.randint(1, 10 ** 6),
                "nmax": _log_int(rng, 2000, 20000), "prec": "bf16_mixed"}
    n = _log_int(rng, 20000, 400000)
    return {"kind": kind, "data": "curved", "n": n, "m": _log_int(rng, 128, 4096), "k": rng.randint(10, 64),
            "dtype": "bf16", "rows": _log_int(rng, 2000, min(n, 20000)), "prec": "bf16_mixed"}


# ---- inputs -------------------------------------------------------------------
def _gen(seed, tag=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + tag) % (1 << 62))
    return g


def _frame(m, d, g):
    return torch.linalg.qr(torch.randn(m, d, generator=g, device=DEV, dtype=torch.float64))[0].float()


def _mlp(z, widths, g, bias=0.1):
    h = z
    for i, w in enumerate(widths):
        a = torch.randn(h.shape[1], w, generator=g, device=DEV) / math.sqrt(h.shape[1])
        h = h @ a + bias * torch.randn(w, generator=g, device=DEV)
        if i + 1 < len(widths):
            h = torch.tanh(h)
    return h


def _points(data, n, m, dtype, seed, d=None):
    """n x m points of one of ``synth``'s recipes, drawn on the GPU."""
    g = _gen(seed, 1)
    if data == "sphere":
        u = torch.randn(n, 3, generator=g, device=DEV)
        u /= u.norm(dim=1, keepdim=True)
        x = u @ _frame(m, 3, g).T + 0.01 * torch.randn(n, m, generator=g, device=DEV)
    elif data == "decoder":
        x = _mlp(torch.randn(n, 10, generator=g, device=DEV), [64, 128, m], g)
    elif data == "mlp":
        x = _mlp(torch.randn(n, d or 8, generator=g, device=DEV), [64, m], g)
        x = x + 0.01 * torch.randn(n, m, generator=g, device=DEV)
    elif data == "sparse":
        mask = torch.rand(10, m, generator=g, device=DEV) < 0.18
        mu = torch.where(mask, 0.25 + 0.75 * torch.rand(10, m, generator=g, device=DEV),
                         torch.full((10, m), -0.3, device=DEV))
        of = torch.randint(0, 10, (n,), generator=g, device=DEV)
        x = (mu[of] + 0.15 * torch.randn(n, m, generator=g, device=DEV)).clamp_(0.0, 1.0)
    elif data == "curved":
        patches = max(1, min(32, n // 2000))
        x = torch.empty(n, m, dtype=torch.bfloat16, device=DEV)
        perm = torch.randperm(n, generator=g, device=DEV)
        cut = [n * c // patches for c in range(patches + 1)]
        dl = min(8, m - 1)
        for c in range(patches):
            rows = perm[cut[c]:cut[c + 1]]
            a = torch.triu(torch.randn(dl, dl, generator=g, device=DEV))
            a = a + torch.triu(a, 1).T
            f = _frame(m, dl + 1, g)
            o = 0.5 * torch.randn(m, generator=g, device=DEV)
            u = 2 * torch.rand(len(rows), dl, generator=g, device=DEV) - 1
            h = 0.5 * ((u @ a) * u).sum(1, keepdim=True)
            blk = torch.cat([u, h], 1) @ f.T
            blk += o
            blk += 0.005 * torch.randn(len(rows), m, generator=g, device=DEV)
            x[rows] = blk.to(torch.bfloat16)
    else:
        raise ValueError(data)
    return x.to(torch.bfloat16 if dtype == "bf16" else torch.float32).contiguous()


def _neighbours(x, k):
    """The k nearest other rows of every row (FP32 distances), int32."""
    x = x.float()
    c = x - x.mean(0)
    sq = (c * c).sum(1)
    n = x.shape[0]
    out = torch.empty(n, k, dtype=torch.int32, device=x.device)
    step = max(64, (1 << 28) // n)
    for a in range(0, n, step):
        b = min(n, a + step)
        d = sq[None, :] - 2.0 * (c[a:b] @ c.T)
        d[torch.arange(b - a, device=x.device), torch.arange(a, b, device=x.device)] = math.inf
        out[a:b] = d.topk(k, largest=False).indices.int()
    return out


def _set_shapes(case):
    r = np.random.default_rng(case["shape_seed"])
    out = []
    for _ in range(case["sets"]):
        out.append((int(r.integers(500, case["nmax"] + 1)), int(r.choice([64, 128, 256, 512, 1024])),
                    int(r.integers(10, 65)), int(r.integers(2, 17))))
    return out


def prepare(case, seed):
    st = {"case": case, "ctx": api.context(0)}
    if case["kind"] == "batched":
        shapes = _set_shapes(case)
        st["Xs"] = [_points("mlp", n, m, "f32", seed * 131 + i, d) for i, (n, m, k, d) in enumerate(shapes)]
        st["ks"] = [s[2] for s in shapes]
        return st
    st["X"] = _points(case["data"], case["n"], case["m"], case["dtype"], seed)
    if case["kind"] in ("curvature", "grad"):
        st["idx"] = _neighbours(st["X"], case["k"])
    if case["kind"] == "grad":
        st["X"].requires_grad_(True)
        st["dk"] = torch.rand(case["n"], generator=_gen(seed, 2), device=DEV) + 0.5
    return st


def run(st):
    c, ctx = st["case"], st["ctx"]
    kind = c["kind"]
    if kind == "knn":
        idx, dist = ctx.mecuco_knn(st["X"], c["k"], precision=c["prec"], return_dist=True)
        return {"idx": idx, "dist": dist}
    if kind == "curvature":
        return ctx.mecuco_curvature(st["X"], c["k"], idx=st["idx"], variant=c["variant"], precision=c["prec"],
                                    return_lambda=True)
    if kind == "exact":
        return {"kappa": ctx.curvature_auto(st["X"], c["k"], precision=c["prec"])}
    if kind == "grad":
        kappa = autograd.curvature(st["X"], st["idx"], c["k"], c["variant"])
        dx, = torch.autograd.grad(kappa, st["X"], st["dk"])
        return {"kappa": kappa.detach(), "dX": dx}
    if kind == "batched":
        return ctx.mecuco_curvature_batched(st["Xs"], st["ks"], precision=c["prec"])
    # a shard of query rows against every point
    idx = ctx.mecuco_knn_range(st["X"], c["k"], 0, c["rows"], precision=c["prec"])
    kappa = ctx.mecuco_curvature_range(st["X"], c["k"], 0, c["rows"], idx=idx, precision=c["prec"])
    return {"idx": idx, "kappa": kappa}


# ---- work ---------------------------------------------------------------------
def _point_flops(m, k):
    """Gram, distinct third moments of a patch, and an eigensolve of order k."""
    return k * (k + 1) * m + k * (k + 1) * (k + 2) // 6 * 2 * m + 9 * k ** 3


def work(case):
    kind = case["kind"]
    if kind == "batched":
        b = f = 0
        for n, m, k, _ in _set_shapes(case):
            b += 4 * n * m + 4 * n
            f += 2 * n * n * m + n * _point_flops(m, k)
        return {"bytes": b, "flops": f}
    n, m, k = case["n"], case["m"], case["k"]
    e = 2 if case["dtype"] == "bf16" else 4
    x = n * m * e
    if kind == "knn":
        return {"bytes": x + 8 * n * k, "flops": 2 * n * n * m}
    if kind == "curvature":
        return {"bytes": x + 4 * n * k + 4 * n + 4 * n * k, "flops": n * _point_flops(m, k)}
    if kind == "exact":
        return {"bytes": x + 4 * n, "flops": 2 * n * n * m + n * (k * m * (m + 1) + 9 * m ** 3 + 2 * m ** 3)}
    if kind == "grad":
        # forward moments twice (the backward recomputes them) and the adjoint's
        # contraction of every patch column with the third-moment gradient
        return {"bytes": 2 * x + 4 * n * k + 8 * n + 4 * n * m, "flops": n * (2 * _point_flops(m, k) + k ** 3 * m)}
    r = case["rows"]
    return {"bytes": x + 4 * r * k + 4 * r, "flops": 2 * r * n * m + r * _point_flops(m, k)}


# ---- FP64 values --------------------------------------------------------------
def _knn64(x, k, want_idx=False):
    """Exact neighbours: FP32 preselection of k + 32, then FP64 distances."""
    n = x.shape[0]
    pre = _neighbours(x, min(n - 1, k + 32)).long()
    x64 = x.double()
    dist = torch.empty(n, k, dtype=torch.float64, device=x.device)
    idx = torch.empty(n, k, dtype=torch.int64, device=x.device)
    step = max(1, (1 << 28) // (pre.shape[1] * x.shape[1]))
    for a in range(0, n, step):
        b = min(n, a + step)
        d = (x64[pre[a:b]] - x64[a:b, None, :]).square().sum(2)
        v, o = d.sort(dim=1, stable=True)
        dist[a:b] = v[:, :k]
        idx[a:b] = pre[a:b].gather(1, o[:, :k])
    return (idx, dist) if want_idx else dist


def _fast64(x, idx, variant, need_lambda=False, rank_tol=2.0 ** -52):
    """Fast-mode curvature of every row of idx, term by term."""
    n, k = idx.shape
    m = x.shape[1]
    kap = torch.empty(n, dtype=torch.float64, device=x.device)
    lam_out = torch.zeros(n, k, dtype=torch.float64, device=x.device)
    step = max(1, (1 << 27) // (k * m))
    for a in range(0, n, step):
        xc = x[idx[a:a + step].long()].double()
        xc = xc - xc.mean(1, keepdim=True)
        kap[a:a + step], lam_out[a:a + step] = _fast_terms(xc, variant)
    return (kap, lam_out) if need_lambda else kap


def _fast_terms(xc, variant):
    b, k, m = xc.shape
    p = min(k - 1, m)
    w, u = torch.linalg.eigh(xc @ xc.transpose(1, 2))
    w, u = w.flip(1)[:, :p], u.flip(2)[:, :, :p]
    v = xc.transpose(1, 2) @ (u / w.sqrt()[:, None, :])  # b x m x p
    km1 = k - 1
    tau = w.sum(1) / km1
    av = xc @ v.square()
    t_range = av.square().sum((1, 2)) / km1
    dp = 1.0 - v.square().sum(2)
    t_a = (xc @ dp[:, :, None]).square().sum((1, 2)) / km1
    gt2 = torch.zeros_like(tau)
    for r in range(p):
        s = (xc * v[:, None, :, r]) @ v[:, :, r:]
        gt2 = gt2 + 2.0 * s.square().sum((1, 2)) - s[:, :, 0].square().sum(1)
    q = m - p
    t_null = torch.zeros_like(tau)
    if q > 0:
        if variant == "haar":
            mid = (xc.square().sum(1) * (1.0 - dp)).sum(1) / km1
            t_null = (t_a + 2.0 * (tau - 2.0 * mid + gt2 / km1)) / (q + 2)
        else:
            t_null = (t_a + 2.0 * (-tau + gt2 / km1)) / q
    lam = torch.zeros(b, k, dtype=xc.dtype, device=xc.device)
    lam[:, :p] = w / km1
    return (0.5 * (t_range + t_null) + 0.5 * tau).abs(), lam


def _exact_mode64(x, idx):
    n, k = idx.shape
    out = torch.empty(n, dtype=torch.float64, device=x.device)
    for a in range(0, n, 4096):
        xc = x[idx[a:a + 4096]].double()
        xc = xc - xc.mean(1, keepdim=True)
        v, w = torch.linalg.eigh(xc.transpose(1, 2) @ xc / (k - 1))
        c = w.transpose(1, 2) @ w.square()
        out[a:a + 4096] = (0.5 * (v * c.square().sum(2)).sum(1) + 0.5 * v.sum(1)).abs()
    return out


def _cost64(n, m, k, search):
    """Rough FP64 operations of exact() for one dataset."""
    return n * (k * m * k * k + 40 * k ** 3 + (3 * (k + 32) * m if search else 0))


def exact(case, seed):
    kind = case["kind"]
    if kind == "whole":
        return None
    if kind == "batched":
        shapes = _set_shapes(case)
        if sum(_cost64(n, m, k, True) for n, m, k, _ in shapes) > 8e12:
            return None
        out = []
        for i, (n, m, k, d) in enumerate(shapes):
            if k - 1 > m:
                out.append(None)
                continue
            x = _points("mlp", n, m, "f32", seed * 131 + i, d)
            idx, _ = _knn64(x, k, True)
            out.append(_fast64(x, idx, "literal"))
        return out
    n, m, k = case["n"], case["m"], case["k"]
    x = _points(case["data"], n, m, case["dtype"], seed)
    if kind == "knn":
        return {"idx": None, "dist": _knn64(x, k)}
    if kind == "exact":
        idx, _ = _knn64(x, k, True)
        return {"kappa": _exact_mode64(x, idx)}
    idx = _neighbours(x, k)
    if kind == "curvature":
        if _cost64(n, m, k, False) > 8e12:
            return None
        kap, lam = _fast64(x, idx, case["variant"], need_lambda=True)
        return {"kappa": kap, "lambda": lam}
    # grad: autograd in FP64 through the same terms, neighbour lists fixed
    dk = (torch.rand(n, generator=_gen(seed, 2), device=DEV) + 0.5).double()
    dx = torch.zeros(n, m, dtype=torch.float64, device=DEV)
    kap = torch.empty(n, dtype=torch.float64, device=DEV)
    step = max(1, (1 << 24) // (k * m))
    for a in range(0, n, step):
        rows = idx[a:a + step].long()
        xp = x[rows].double().requires_grad_(True)
        kk, _ = _fast_terms(xp - xp.mean(1, keepdim=True), case["variant"])
        g, = torch.autograd.grad(kk, xp, dk[a:a + step])
        kap[a:a + step] = kk.detach()
        dx.index_add_(0, rows.reshape(-1), g.reshape(-1, m))
    return {"kappa": kap, "dX": dx}
