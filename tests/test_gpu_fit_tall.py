"""Fits of large vocabularies, whose product with the subspace has too many row tiles to
be split over the terms, with words that never occur."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("V,D", [(9800, 120), (19500, 8)])
def test_fit_of_a_large_vocabulary(lib, V, D):
    sparse = pytest.importorskip("scipy.sparse")
    from scipy.sparse.linalg import LinearOperator, eigsh

    a0 = 1.0
    # per word its own documents (the word three times, every second one with the next word once): many for the first
    # D words, two for the others, none for every tenth of those (nor is it a next word)
    n = np.where(np.arange(V) < D, np.geomspace(400, 100, V).astype(int), 2)
    n[D + 5::10] = 0
    word = np.repeat(np.arange(V), n)
    nxt = (word + 1) % V
    pair = (np.arange(len(word)) % 2 == 0) & (n[nxt] > 0)
    lo, hi = np.minimum(word, nxt), np.maximum(word, nxt)
    idx = np.where(pair[:, None], np.stack([lo, hi], 1), np.stack([word, np.full_like(word, -1)], 1)).ravel()
    cnt = np.where(pair[:, None], np.stack([np.where(word < nxt, 3, 1), np.where(word < nxt, 1, 3)], 1), 3).ravel()
    keep = idx >= 0
    idx, cnt = idx[keep], cnt[keep]
    indptr = np.concatenate([[0], np.cumsum(1 + pair)])
    t = lib.TLDA(V, D, alpha0=a0, max_batch=64)
    t.fit([lib.DeviceCSR.from_arrays(indptr, idx, cnt, V)])
    W, m1, ev = t.get_whitening()
    t.close()
    W = W.cpu().numpy().astype(np.float64)
    F = sparse.csr_matrix((cnt.astype(float), idx, indptr), shape=(len(word), V))
    L, c = np.asarray(F.sum(axis=1)).ravel(), np.asarray(F.sum(axis=0)).ravel()
    assert (c == 0).sum() == (n == 0).sum() > 0
    M1, P = c / L.sum(), F.T @ F - sparse.diags(c)

    def M2(x):
        return (a0 + 1) * (P @ x) / (L * (L - 1)).sum() - a0 * np.multiply.outer(M1, M1 @ x)

    lam = np.sort(eigsh(LinearOperator((V, V), matvec=lambda x: M2(x.ravel())), k=D, which="LA", tol=1e-12)[0])[::-1]
    # as at the widest models: an FP32 subspace, FP64 Ritz pairs, W rounded to FP32
    assert np.abs(ev - lam).max() <= (2.0 ** -24 * np.sqrt(V) * 64) ** 2 * lam[0]
    assert np.abs(W.T @ M2(W) - np.eye(D)).max() <= 2.0 ** -24 * 4 * np.sqrt(lam[0] / lam[-1])
    assert np.abs(m1.cpu().numpy() - W.T @ M1).max() <= 2.0 ** -22 * np.abs(W).max()
