"""Edges of the size-dependent kernel paths, against the fp64 oracle: the smallest and largest of
each path's range, remainders of its tiles, and both sides of each dispatch rule."""

import numpy as np
import pytest
import torch

from oracle import loca_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2608_03020_gb300 import _build

    _build.build()
    from paper_2608_03020_gb300 import loca

    loca.lib()
    return loca


def _np(t):
    return t.detach().double().cpu().numpy()


def _rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def _dev(a, dtype=torch.float32):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dtype)


@pytest.mark.parametrize("L,N,d,C,r,batches", [
    (2, 65, 40, 2, 3, 2),       # one partial tile in every direction, U columns padded to 32
    (1, 130, 8456, 4, 5, 1),    # two column ranges of S, the second ragged and without 4-D loads
    (2, 70, 264, 8, 17, 2),     # U columns padded to 64, an 8-column last tile
])
def test_factored_cross_product(lc, L, N, d, C, r, batches):
    """cross = Q^T ((E P)^T X): U's two bf16 parts carry 2^-17 = 7.6e-6 of each entry, the sums
    over a few hundred tokens and over r are fp32, so 2e-5 of the exact product."""
    rng = np.random.default_rng(d)
    gram, cross = (torch.full((L, d, d), float("nan"), device="cuda") for _ in range(2))
    P = rng.normal(0, 1, (L, C, r)).astype(np.float32)
    Q = rng.normal(0, 1, (L, r, d)).astype(np.float32)
    alpha = np.linspace(0.5, -1.0, L).astype(np.float32)
    ref = np.zeros((L, d, d))
    gref = np.zeros((L, d, d))
    for b in range(batches):
        X = torch.from_numpy(rng.standard_normal((L, N, d)).astype(np.float32)).to(torch.bfloat16)
        E = rng.standard_normal((N, C)).astype(np.float32)
        lc.loca_gram_cross_fused(X.to("cuda"), _dev(E), _dev(P), _dev(Q), _dev(alpha), gram, cross, zero_first=b == 0)
        Xn = X.double().numpy()
        T, _ = O.feedback_targets(E, P, Q)
        for l in range(L):
            ref[l] += float(alpha[l]) * (T[l].T @ Xn[l])
            gref[l] += Xn[l].T @ Xn[l]
    torch.cuda.synchronize()
    assert lc.loca_device_status() == 0
    assert _rel(_np(cross), ref) <= 2e-5
    assert _rel(_np(gram), gref) <= 2e-5


@pytest.mark.parametrize("N,C", [(1, 1), (513, 16), (1500, 17), (700, 64)])
def test_targets_sq_entry_groups(lc, N, C):
    """One thread group per E^T E entry up to C = 16, several entries per thread above: fp64 sums of
    fp64 products, M = Q Q^T from fp32 runs of 32 products (32 * 2^-24 = 2e-6)."""
    rng = np.random.default_rng(N)
    E = rng.standard_normal((N, C)).astype(np.float32)
    P = rng.standard_normal((2, C, 7)).astype(np.float32)
    Q = rng.standard_normal((2, 7, 100)).astype(np.float32)
    tsq = torch.empty((2,), dtype=torch.float64, device="cuda")
    lc.loca_targets_sq(_dev(E), _dev(P), _dev(Q), tsq)
    _, ref = O.feedback_targets(E, P, Q)
    assert np.allclose(_np(tsq), ref, rtol=2e-6, atol=0)


@pytest.mark.parametrize("L,N,d", [(1, 1, 1), (2, 63, 33), (1, 64, 32), (3, 257, 65), (1, 2000, 31), (2, 300, 250)])
def test_fp32_statistics_token_split(lc, L, N, d):
    """The fp32-input statistics at every cluster size (1 to 8 token ranges, ragged and empty ones) and
    tile remainders: fp64 sums, so the fp32 rounding of the exact result (2^-24 = 6e-8 of each entry)
    and, accumulated over two batches, one more."""
    rng = np.random.default_rng(N * 7 + d)
    gram, cross = (torch.full((L, d, d), float("nan"), device="cuda") for _ in range(2))
    alpha = np.linspace(0.5, -1.0, L).astype(np.float32)
    g_ref, c_ref = np.zeros((L, d, d)), np.zeros((L, d, d))
    for b in range(2):
        X, T = (rng.standard_normal((L, N, d)).astype(np.float32) for _ in range(2))
        lc.loca_gram_cross(_dev(X), _dev(T), _dev(alpha), gram, cross, zero_first=b == 0)
        for l in range(L):
            x, t = X[l].astype(np.float64), T[l].astype(np.float64)
            g_ref[l] += x.T @ x
            c_ref[l] += float(alpha[l]) * (t.T @ x)
    assert _rel(_np(gram), g_ref) <= 1.2e-7 and _rel(_np(cross), c_ref) <= 1.2e-7
    assert torch.equal(gram, gram.transpose(1, 2))


@pytest.mark.parametrize("Np,m,d,L,r", [
    (33, 1, 1, 1, 1),        # one run and a remainder, one column
    (1025, 8, 131, 2, 3),    # 4 columns per lane, odd width (scalar loads), two token ranges
    (2100, 9, 130, 1, 9),    # 2 columns per lane (16-byte rows fail, 8-byte rows load)
    (1500, 17, 64, 2, 5),    # one column per lane
    (1100, 33, 70, 1, 6),    # two groups of sums
])
def test_calibration_and_alignment_paths(lc, Np, m, d, L, r):
    """The fit's sums are fp32 over 32 tokens and exact to 2^-48 beyond, its solves fp64: the product
    P Q within 1e-5 (fp32 inputs, beta = 1e-3 of the mean eigenvalue, decaying planted spectrum); the
    diagnostic on the fitted factors within 1e-5."""
    rng = np.random.default_rng(Np + m)
    E = rng.standard_normal((Np, m)).astype(np.float32)
    planted = [(rng.standard_normal((m, r)) * 0.7 ** np.arange(r)) @ rng.standard_normal((r, d)) for _ in range(L)]
    G = np.stack([E @ M + 0.05 * rng.standard_normal((Np, d)) for M in planted]).astype(np.float32)
    r = min(r, m, d)
    beta = 1e-3 * float(np.sum(E.astype(np.float64) ** 2)) / m
    P, Q = torch.empty((L, m, r), device="cuda"), torch.empty((L, r, d), device="cuda")
    sigma, alpha = torch.empty((L, r), device="cuda"), torch.empty((L,), dtype=torch.float64, device="cuda")
    lc.loca_calib_fit(_dev(E), _dev(G), beta, r, P, Q, sigma=sigma)
    lc.loca_alignment(_dev(E), _dev(G), P, Q, alpha)
    torch.cuda.synchronize()
    assert lc.loca_device_status() == 0
    P_ref, Q_ref, s_ref, _ = O.calib_fit(E, G, beta, r)
    for l in range(L):
        assert _rel(_np(P[l]) @ _np(Q[l]), P_ref[l] @ Q_ref[l]) <= 1e-5
    assert _rel(_np(sigma), s_ref) <= 1e-5
    ref = O.alignment(E, _np(P), _np(Q), G)
    assert np.max(np.abs(_np(alpha) - ref)) <= 1e-5


@pytest.mark.parametrize("Np,m,d,L,r,ell,q", [
    (300, 130, 70, 10, 4, 8, 1),    # columns divided over the SMs (one each), 8-wide streams of G
    (200, 65, 129, 26, 3, 6, 1),    # two columns a CTA; ell no multiple of 4: tiled G^T products
    (257, 192, 101, 8, 8, 20, 0),   # 32-wide streams over 20-column blocks, scalar loads, fp64 solves only
    (150, 70, 80, 3, 2, 4, 2),      # few columns: step-by-step solves
    (150, 70, 80, 3, 8, 40, 1),     # 64-column tiles for one block's products
])
def test_wide_calibration_paths(lc, Np, m, d, L, r, ell, q):
    """P Q against the oracle's same steps: fp32 runs of 32 products, exact to 2^-48 beyond, fp64 solves
    where they count; planted rank r with a decaying spectrum and 1% noise, so 1e-5."""
    rng = np.random.default_rng(Np + ell)
    E = (rng.standard_normal((Np, m)) * rng.lognormal(0, 0.3, m)).astype(np.float32)
    G = np.empty((L, Np, d), dtype=np.float32)
    for l in range(L):
        clean = (E @ (rng.standard_normal((m, r)) * 0.7 ** np.arange(r))) @ rng.standard_normal((r, d))
        G[l] = clean + 0.01 * np.sqrt(np.mean(clean ** 2)) * rng.standard_normal((Np, d))
    Om = rng.standard_normal((d, ell)).astype(np.float32)
    beta = 1e-3 * float(np.sum(E.astype(np.float64) ** 2)) / m
    P, Q = torch.empty((L, m, r), device="cuda"), torch.empty((L, r, d), device="cuda")
    sigma, alpha = torch.empty((L, r), device="cuda"), torch.empty((L,), dtype=torch.float64, device="cuda")
    lc.loca_calib_fit_rsvd(_dev(E), _dev(G), beta, r, _dev(Om), q, P, Q, sigma=sigma)
    lc.loca_alignment(_dev(E), _dev(G), P, Q, alpha)
    torch.cuda.synchronize()
    assert lc.loca_device_status() == 0
    P_ref, Q_ref, s_ref = O.calib_fit_rsvd(E, G, beta, r, Om, q)
    for l in range(L):
        assert _rel(_np(P[l]) @ _np(Q[l]), P_ref[l] @ Q_ref[l]) <= 1e-5
    assert _rel(_np(sigma), s_ref) <= 1e-5
    assert np.max(np.abs(_np(alpha) - O.alignment(E, _np(P), _np(Q), G))) <= 1e-5
