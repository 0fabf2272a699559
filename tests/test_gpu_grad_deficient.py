"""The gradient of patches with a null space (fewer columns than neighbours, a low-rank
set, copies): the adjoint's formulas over the range eigenpairs in FP64.  The null
vectors have eigenvalues of rounding noise, any two of which are a gap apart."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _adjoint64(x, idx, haar):
    """d(sum K)/dX by the adjoint's formulas (range eigenpairs from an SVD of each patch)."""
    k, m = idx.shape[1], x.shape[1]
    out = torch.zeros_like(x)
    km1 = k - 1
    for rows in idx.long():
        xc = x[rows] - x[rows].mean(0)
        u, s, _ = torch.linalg.svd(xc, full_matrices=True)
        lam = torch.zeros(k, dtype=x.dtype)
        lam[:len(s)] = s.square()
        if float(lam[0]) == 0.0:
            continue
        p = min(k - 1, m, int((lam > k * m * 2.0 ** -52 * lam[0]).sum()))
        q = m - p
        c = (1.0 / (q + 2) if haar else 1.0 / q) if q > 0 else 0.0
        w = u[:, :p] / s[:p]
        M = torch.einsum("ja,ra,ta->jrt", xc, xc, xc)
        S = torch.einsum("rl,jrt,tu->jlu", w, M, w)
        A = torch.diagonal(S, dim1=1, dim2=2)
        xd = xc.sum(1) - A.sum(1)
        cw = xc.square().sum(0)
        Q = (xc * cw) @ xc.T
        tau, gt2 = lam[:p].sum() / km1, S.square().sum() / km1
        t_b = tau - 2.0 * torch.einsum("rl,rt,tl->", w, Q, w) / km1 + gt2 if haar else gt2 - tau
        t_null = (xd.square().sum() / km1 + 2.0 * t_b) * c
        sgn = torch.sign(0.5 * (A.square().sum() / km1 + t_null) + 0.5 * tau)
        dS = 2.0 * sgn * c / km1 * S + torch.diag_embed(sgn * (A - c * xd[:, None]) / km1)
        dM = torch.einsum("rl,jlu,tu->jrt", w, dS, w)
        dW = 2.0 * torch.einsum("jrt,tl,jlu->ru", M, w, dS)
        dtau = sgn * (0.5 + (c if haar else -c))
        if haar:
            dh = -2.0 * sgn * c / km1
            dQ = dh * w @ w.T
            dW = dW + 2.0 * dh * Q @ w
        du = torch.zeros(k, k, dtype=x.dtype)
        du[:, :p] = dW / s[:p]
        ds2 = torch.zeros(k, dtype=x.dtype)
        ds2[:p] = dtau / km1 - 0.5 * (u[:, :p] * dW).sum(0) / s[:p] ** 3
        gap = lam[None, :] - lam[:, None]
        f = torch.where(gap != 0, 1.0 / gap, torch.zeros_like(gap))
        f[:, p:] = 0.0
        f.fill_diagonal_(0.0)
        g = u @ (torch.diag(ds2) + f * (u.T @ du)) @ u.T
        d = (g + g.T) @ xc + (sgn * c * xd / km1)[:, None]
        C = dM + dM.permute(1, 0, 2) + torch.einsum("tir->irt", dM)
        d = d + torch.einsum("irt,ra,ta->ia", C, xc, xc)
        if haar:
            d = d + 2.0 * cw * (dQ @ xc) + 2.0 * xc * (xc * (dQ @ xc)).sum(0)
        out.index_add_(0, rows, d - d.mean(0))
    return out


def _set(kind, n, m):
    g = torch.Generator().manual_seed(n + m)
    r = lambda *s: torch.randn(*s, generator=g, dtype=torch.float64)
    if kind == "full":
        return r(n, m)
    if kind == "lowrank":
        return r(n, 3) @ r(3, m)
    return r((n + 3) // 4, m).repeat_interleave(4, 0)[:n]  # copies


@pytest.mark.parametrize("variant", ["literal", "haar"])
@pytest.mark.parametrize("kind,n,m,k", [("full", 70, 1, 12), ("full", 70, 2, 17), ("full", 60, 7, 30),
                                        ("full", 60, 16, 41), ("lowrank", 65, 300, 19), ("lowrank", 50, 40, 33),
                                        ("copies", 60, 33, 32), ("copies", 60, 150, 20)])
def test_gradient_with_a_null_space(kind, n, m, k, variant):
    from paper_2606_06329_gb300 import api
    X = _set(kind, n, m).float()
    with api.Context(0) as c:
        idx = c.mecuco_knn(X.cuda(), k)
        got = c.mecuco_curvature_backward(X.cuda(), k, idx, torch.ones(n, device="cuda"), variant=variant)
        assert c.mecuco_get_last_status() == 0
    ref = _adjoint64(X.double(), idx.cpu(), variant == "haar")
    err = float((got.cpu().double() - ref).norm() / ref.norm())
    print(f"{kind} n={n} m={m} k={k} {variant}: {err:.1e}")
    assert err < 1e-3  # the gradient's target on its norm
