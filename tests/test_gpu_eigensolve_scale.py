"""The eigensolve of the online whitening at scales beyond FP32's range: a power of
two over the statistics is one over the whitening."""
import numpy as np
import pytest

from .test_gpu_eigensolve import D, V, _planted

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("r", [32, 130])
@pytest.mark.parametrize("exp", [-140, -60, 200])
def test_scale(lib, r, exp):
    U, Om, lam, _, _, _ = _planted(r)
    Z = (U * lam) @ (U.T @ Om) * 500.0  # alpha0 = 1, S2 = 1000, no words counted: M2 = U lam U^T
    t = lib.TLDA(V, D, alpha0=1.0, max_batch=64)
    t.online_begin(torch.tensor(Om))
    out = []
    for e in (0, exp):
        t.online_set_sketch(torch.tensor(np.ldexp(Z, e)), torch.zeros(V, dtype=torch.int64), torch.tensor([1, 1000, 0]))
        t.online_whiten()
        W, _, ev = t.get_whitening()
        out.append((np.ldexp(W.cpu().numpy().astype(np.float64), e // 2), np.ldexp(ev, -e)))
    t.close()
    (W0, ev0), (W1, ev1) = out
    bound = 2.0 ** -52 * 64 * r * 1e3  # as alone
    assert np.abs(ev1 - np.sort(lam)[::-1][:D]).max() <= bound
    # eigenvectors to the bound over the gaps of the spectrum, then FP32 rounding
    gap = np.diff(np.sort(lam)).min()
    assert np.abs(W1 - W0).max() <= (2.0 ** -22 + 2 * bound / gap) * np.abs(W0).max()
