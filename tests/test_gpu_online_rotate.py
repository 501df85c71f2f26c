"""Factors carried from a whitening that has no full rank: the Cholesky factor gives up,
the elimination behind it finds no pivot, and the factors stay as they are."""
import numpy as np
import pytest

from .test_gpu_eigensolve import A0, D, V, _planted

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("how", ["zero", "nan"])
def test_singular_previous_whitening(lib, how):
    _, Om, _, C, _, Z = _planted(32)
    rng = np.random.default_rng(1)
    W = rng.standard_normal((V, D)).astype(np.float32)
    W[:, 3] = 0.0
    if how == "nan":
        W[7, 3] = np.nan
    t = lib.TLDA(V, D, alpha0=A0, max_batch=64)
    t.set_whitening(torch.tensor(W), torch.zeros(D))
    t.online_begin(torch.tensor(Om))
    t.online_set_sketch(torch.tensor(Z), torch.tensor(C), torch.tensor([int(C.sum()), 1000, 0]))
    Phi = torch.tensor(rng.standard_normal((D, D)).astype(np.float32), device="cuda")
    before = Phi.cpu().numpy().copy()
    with pytest.raises(lib.TLDAError) as e:
        t.online_whiten(Phi)
    assert e.value.status == lib.ERR_NUMERIC
    assert np.array_equal(Phi.cpu().numpy(), before)
    t.close()
