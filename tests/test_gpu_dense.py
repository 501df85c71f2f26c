"""The FP64 algebra of the moments and of recovery (tensor-core products in exact
slices, panel Cholesky, Jacobi) at the edges of their tiles, against numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _model(V, K, D, W):
    from paper_2511_07809_gb300 import tlda

    t = tlda.TLDA(V, K, dim=D, max_batch=64)
    t.set_whitening(torch.tensor(W, dtype=torch.float32), torch.zeros(D))
    return t


# columns over one, below, at and above a 64-wide tile and a 32-column panel; rows
# below a tile, at odd counts, over several splits of the terms
@pytest.mark.parametrize("V,D,K", [(1, 1, 1), (33, 5, 3), (64, 31, 31), (200, 33, 32), (257, 64, 64), (1000, 65, 65),
                                   (999, 97, 50), (5001, 129, 128), (700, 300, 257), (2048, 512, 511)])
def test_topics_at_tile_edges(V, D, K):
    rng = np.random.default_rng(V + D)
    # orthonormal columns times scales over 2^20, so that the operands' exponents differ
    W = np.linalg.qr(rng.standard_normal((V, D)))[0] * 2.0 ** rng.integers(-10, 11, D)
    W = W.astype(np.float32).astype(np.float64)
    Phi = rng.standard_normal((D, K)).astype(np.float32).astype(np.float64)
    t = _model(V, K, D, W)
    mu, alpha = t.unwhiten_topics(torch.tensor(Phi, dtype=torch.float32, device="cuda"))
    t.close()
    n2 = (Phi ** 2).sum(axis=0)
    # (W^T W)^-1 Phi without squaring the scales: W = Q R
    Q, R = np.linalg.qr(W)
    raw = Q @ np.linalg.solve(R.T, Phi) * n2
    ref = np.maximum(raw, 0.0)
    tot = ref.sum(axis=0)
    ref = ref / np.where(tot > 0, tot, 1.0)
    # W^T W = Q-scaled: after its columns' scales are divided out its condition is 1 to FP32 rounding, and the
    # Cholesky factor, its inverse and the products keep FP64 rounding of terms below 2^20 ||Phi|| each
    bound = 2.0 ** -52 * 64 * D * np.abs(raw).max() / np.where(tot > 0, tot, 1.0).min()
    assert np.abs(mu - ref).max() <= bound, (np.abs(mu - ref).max(), bound)
    a = n2 ** -3.0
    assert np.abs(alpha - a / a.sum()).max() <= 1e-13


def test_topics_of_a_nan_whitening_fail():
    from paper_2511_07809_gb300 import tlda

    W = np.linalg.qr(np.random.default_rng(0).standard_normal((100, 8)))[0]
    W[3, 2] = np.nan
    t = _model(100, 8, 8, W)
    with pytest.raises(tlda.TLDAError) as e:
        t.unwhiten_topics(torch.ones((8, 8), device="cuda"))
    assert e.value.status == tlda.ERR_NUMERIC
    t.close()


# sketch widths around the panels of the Cholesky factor and the tiles of the Jacobi rounds
@pytest.mark.parametrize("r", [32, 34, 64, 66, 130, 258])
def test_online_whitening_at_widths(r):
    from paper_2511_07809_gb300 import tlda

    V, D = 600, 20
    rng = np.random.default_rng(r)
    # statistics with a planted spectrum: M2 of known eigenpairs, alpha0 small so that Z alone carries it
    Om = rng.choice([-1.0, 1.0], (V, r))
    U = np.linalg.qr(rng.standard_normal((V, r)))[0]
    lam = np.geomspace(1.0, 1e-3, r) * np.where(np.arange(r) % 3 == 2, -1.0, 1.0)
    C = rng.integers(1, 100, V)
    T, S2, a0 = int(C.sum()), 1000, 1.0
    M1 = C / T
    P = (U * lam) @ U.T + a0 * np.outer(M1, M1)      # M2 of rank r exactly
    Z = P @ Om * S2 / (a0 + 1.0)
    t = tlda.TLDA(V, D, alpha0=a0, max_batch=64)
    t.online_begin(torch.tensor(Om))
    t.online_set_sketch(torch.tensor(Z), torch.tensor(C), torch.tensor([T, S2, 0]))
    t.online_whiten()
    W, m1, ev = t.get_whitening()
    t.close()
    W = W.cpu().numpy().astype(np.float64)
    top = np.sort(lam)[::-1][:D]
    # rank r = the sketch's width: the single-pass formula gives M2 itself, to FP64 rounding times the
    # conditions of Y (1e3 times that of U^T Omega) and of Q^T Omega
    s = np.linalg.svd(U.T @ Om, compute_uv=False)
    bound = 2.0 ** -52 * 64 * r * 1e3 * (s[0] / s[-1]) ** 2
    assert np.abs(ev - top).max() <= bound, (np.abs(ev - top).max(), bound)
    # W^T M2 W = I: FP32 rounding of W besides that
    G = W.T @ ((U * lam) @ (U.T @ W))
    assert np.abs(G - np.eye(D)).max() <= 1e3 * (2.0 ** -22 + bound)
    assert np.abs(m1.cpu().numpy() - W.T @ M1).max() <= 2.0 ** -22 * np.abs(W).max()
