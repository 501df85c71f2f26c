"""Moments and whitening at the widest models: 512 features take a subspace of 528
columns, the largest order of the dense FP64 kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("D", [496, 497, 512])
def test_fit_at_the_widest_models(lib, D):
    V, a0 = 600, 1.0
    # per word m < D its own documents (m three times, every second one with the next word once), few for the
    # words after: M2's eigenvalues fall by 4 over the first D and by some 20 after them
    n = np.where(np.arange(V) < D, np.geomspace(400, 100, V).astype(int), 4)
    word = np.repeat(np.arange(V), n)
    F = np.zeros((len(word), V))
    F[np.arange(len(word)), word] = 3
    F[np.arange(0, len(word), 2), (word[::2] + 1) % V] += 1
    indptr = np.concatenate([[0], np.cumsum((F > 0).sum(axis=1))])
    d, m = np.nonzero(F)
    t = lib.TLDA(V, D, alpha0=a0, max_batch=64)
    t.fit([lib.DeviceCSR.from_arrays(indptr.astype(np.int32), m.astype(np.int32), F[d, m].astype(np.int32), V)])
    W, m1, ev = t.get_whitening()
    t.close()
    W = W.cpu().numpy().astype(np.float64)
    L = F.sum(axis=1)
    M1 = F.sum(axis=0) / L.sum()
    M2 = (a0 + 1) * (F.T @ F - np.diag(F.sum(axis=0))) / (L * (L - 1)).sum() - a0 * np.outer(M1, M1)
    lam = np.linalg.eigvalsh(M2)[::-1][:D]
    # the subspace is found in FP32 (an angle of some 2^-24 sqrt(V) times the spread of the spectrum, squared in
    # the Ritz values), the Ritz pairs in FP64
    assert np.abs(ev - lam).max() <= (2.0 ** -24 * np.sqrt(V) * 64) ** 2 * lam[0]
    # W^T M2 W = I: the columns of W rounded to FP32, each way
    G = W.T @ M2 @ W
    assert np.abs(G - np.eye(D)).max() <= 2.0 ** -24 * 4 * np.sqrt(lam[0] / lam[-1])
    assert np.abs(m1.cpu().numpy() - W.T @ M1).max() <= 2.0 ** -22 * np.abs(W).max()
