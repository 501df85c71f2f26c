"""Steps over a vocabulary that is too large for a block's bitmap of touched words, with a
word that every document holds, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import tlda_oracle as O

from . import _cases as C
from .test_gpu_by_word import _corpus, _model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [131072, 131073, 200001])
@pytest.mark.parametrize("precision,loss,tol", [("fp32", False, 1e-5), ("fp32", True, 1e-5), ("bf16", False, 2e-2)])
def test_step(lib, V, precision, loss, tol):
    rng = np.random.default_rng(V)
    K = 5
    c = _corpus(rng, V, list(rng.integers(3, 40, 300)), 1.0)
    t, W, m1 = _model(lib, rng, V, K, K, precision=precision)
    P0 = (rng.standard_normal((K, K)) / np.sqrt(K)).astype(np.float32)
    Phi = torch.tensor(P0, device="cuda")
    grad = torch.empty_like(Phi)
    dev = lib.DeviceCSR.from_corpus(c)
    for _ in range(2):  # the second step starts from what the first one left behind
        t.cp_step(dev, Phi, 0.0, grad=grad, want_loss=loss)
    t.sync()
    g = O.cp_grad_implicit(c.indptr, c.indices, c.counts, V, W, m1, P0.astype(np.float64), 1.5, 0.0)
    assert C.rel(grad.cpu().numpy(), g["grad"]) < tol
    t.close()
