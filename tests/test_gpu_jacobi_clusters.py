"""The eigensolves and their refinements on Grams of prescribed spectra: clusters of
eigenvalues with relative gaps from 2^-4 to 2^-20, at several magnitudes (192 columns:
the register-resident form; 127: the two-sided sweeps).
The patches' columns are Hadamard vectors times BF16 numbers, so the Gram is known to
FP32 accumulation.  Eigenvectors inside a cluster are as good as the gap lets them be;
orthogonality, residuals and eigenvalues are not allowed that."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _hadamard(k):
    h = np.ones((1, 1))
    while h.shape[0] < k:
        h = np.block([[h, h], [h, -h]])
    return h


def _bf16(v):
    from paper_2606_06329_gb300 import synth
    return synth.bf16_bits_to_f32(synth.f32_to_bf16_bits(np.asarray(v, np.float32))).astype(np.float64)


def _patches(k, m, gap, nclusters, count, seed):
    """count patches of k points (m columns): k - 1 eigenvalues in nclusters clusters a
    factor of 8 apart, relative gap `gap` inside."""
    rng = np.random.default_rng(seed)
    h = _hadamard(k)[:, 1:]
    which = np.sort(rng.integers(0, nclusters, k - 1))
    pos = np.concatenate([np.arange((which == c).sum()) for c in range(nclusters)])
    scale = 2.0 ** (-1.5 * which)
    scale = _bf16(scale)
    X = np.zeros((count, k, m))
    for p in range(count):
        rows, cols = rng.permutation(k), rng.permutation(m)
        sign = rng.choice([-1.0, 1.0], k - 1)
        second = _bf16(scale * np.sqrt(gap * pos))
        X[p][:, cols[:k - 1]] = h[rows] * (sign * scale)
        X[p][:, cols[k - 1:2 * k - 2]] = h[rows] * second
    return X


@pytest.mark.parametrize("m", [127, 192])
@pytest.mark.parametrize("k", [16, 32, 64])
@pytest.mark.parametrize("nclusters", [1, 4])
@pytest.mark.parametrize("log_gap", [-4, -8, -12, -16, -20])
def test_clustered_spectra(m, k, nclusters, log_gap):
    from paper_2606_06329_gb300 import api
    count = 40
    P = _patches(k, m, 2.0 ** log_gap, nclusters, count, 100 * k + nclusters - log_gap)
    X = P.reshape(count * k, m)
    idx = (np.arange(count * k) // k * k)[:, None] + np.arange(k)[None, :]
    with api.Context(0) as c:
        o = c.mecuco_curvature(torch.from_numpy(X.astype(np.float32)).cuda(), k,
                               idx=torch.from_numpy(idx.astype(np.int32)).cuda(), precision="bf16_mixed",
                               return_U=True, return_s=True)
        torch.cuda.synchronize()
        assert c.mecuco_get_last_status() == 0
    U = o["U"].double()[::k].cpu()
    lam = o["s"].double()[::k].cpu().square()
    G = torch.from_numpy(P @ P.transpose(0, 2, 1))
    l1 = torch.linalg.eigvalsh(G)
    top = l1[:, -1]
    orth = float((U.transpose(1, 2) @ U - torch.eye(k)).abs().max())
    res = float(((G @ U - U * lam[:, None, :]).norm(dim=1) / top[:, None]).max())
    val = float(((lam - l1.flip(1)).abs() / top[:, None]).max())
    print(f"m={m} k={k} clusters={nclusters} gap=2^{log_gap}: U^T U - I {orth:.1e}, residual {res:.1e} lambda_1, "
          f"eigenvalues {val:.1e} lambda_1")
    # FP32 columns of 64 entries (2^-24 k^1/2) and the square of a small correction
    assert orth < 2e-6
    # pairs closer than 2^-18 lambda_1 are not told apart, the Gram is within 2^-19
    assert res < 2.0 ** -17
    assert val < 2.0 ** -17


@pytest.mark.parametrize("k", [13, 37, 64])
@pytest.mark.parametrize("log_gap", [-4, -8, -12, -16, -20])
def test_rotation_of_the_plain_form(k, log_gap):
    # general directions: the plain form's U is the rotation (the register-resident
    # solve) times the eigenvectors of a nearly diagonal Gram
    from paper_2606_06329_gb300 import api
    count, m = 40, 150
    rng = np.random.default_rng(k - log_gap)
    X = np.empty((count, k, m))
    for p in range(count):
        q = np.linalg.qr(np.concatenate([np.ones((k, 1)), rng.standard_normal((k, k - 1))], 1))[0][:, 1:]
        v = np.linalg.qr(rng.standard_normal((m, k - 1)))[0]
        s2 = 8.0 ** -rng.integers(0, 3, k - 1) * (1.0 + 2.0 ** log_gap * np.arange(k - 1))
        X[p] = q @ (np.sqrt(s2)[:, None] * v.T)
    X = X.reshape(count * k, m)
    idx = (np.arange(count * k) // k * k)[:, None] + np.arange(k)[None, :]
    with api.Context(0) as c:
        o = c.mecuco_curvature(torch.from_numpy(X.astype(np.float32)).cuda(), k,
                               idx=torch.from_numpy(idx.astype(np.int32)).cuda(), precision="fp32", return_U=True)
        torch.cuda.synchronize()
        assert c.mecuco_get_last_status() == 0
    U = o["U"].double()[::k].cpu()
    orth = float((U.transpose(1, 2) @ U - torch.eye(k)).abs().max())
    print(f"plain k={k} gap=2^{log_gap}: U^T U - I {orth:.1e}")
    # the rotation within 2e-6 as above, the FP32 sweeps' V within 2^-22 a rotation round
    assert orth < 2e-4
