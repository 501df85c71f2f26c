"""A fit whose second moment falls by seven orders of magnitude within the subspace:
the subspace iteration keeps its basis, from any start."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("seed", [0, 1, 3, 4])
def test_fit_of_a_steep_spectrum(lib, seed):
    V, D, a0 = 40, 24, 1.0
    rng = np.random.default_rng(5)
    F = rng.poisson(0.05, (2000, V)) * np.round(10 ** np.linspace(0, 2.9, V))
    F = F[F.sum(axis=1) > 0]
    L = F.sum(axis=1)
    M1 = F.sum(axis=0) / L.sum()
    M2 = (a0 + 1) * (F.T @ F - np.diag(F.sum(axis=0))) / (L * (L - 1)).sum() - a0 * np.outer(M1, M1)
    lam = np.linalg.eigvalsh(M2)[::-1][:D]
    d, m = np.nonzero(F)
    indptr = np.concatenate([[0], np.cumsum((F > 0).sum(axis=1))])
    t = lib.TLDA(V, D, alpha0=a0, seed=seed, max_batch=64)
    t.fit([lib.DeviceCSR.from_arrays(indptr.astype(np.int32), m.astype(np.int32), F[d, m].astype(np.int32), V)])
    W, m1, ev = t.get_whitening()
    t.close()
    W = W.cpu().numpy().astype(np.float64)
    # the subspace of 40 columns is the whole space: the Ritz pairs have FP64 rounding of sums over V terms
    bound = 2.0 ** -52 * 64 * V * lam[0]
    assert np.abs(ev - lam).max() <= bound, (np.abs(ev - lam).max(), bound)
    # W^T M2 W = I: besides that the columns of W rounded to FP32, each way
    G = W.T @ M2 @ W
    assert np.abs(G - np.eye(D)).max() <= 2.0 ** -24 * 4 * np.sqrt(lam[0] / lam[-1]) + bound / lam[-1]
