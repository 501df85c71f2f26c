"""A batch whose first offset is negative: it is reported, and the step after it is right."""
import numpy as np
import pytest
import torch

from oracle import tlda_oracle as O

from . import _cases as C
from .test_gpu_by_word import _corpus, _model

pytestmark = pytest.mark.gpu


# the FP32 form by word, with the loss, and the BF16 form of several kernels
@pytest.mark.parametrize("precision,loss,tol", [("fp32", False, 1e-5), ("fp32", True, 1e-5), ("bf16", False, 2e-2)])
def test_negative_first_offset_leaves_no_trace(lib, precision, loss, tol):
    rng = np.random.default_rng(4)
    V, K = 500, 30
    c = _corpus(rng, V, list(rng.integers(3, 20, 200)), 0.5)
    t, W, m1 = _model(lib, rng, V, K, K, precision=precision)
    P0 = (rng.standard_normal((K, K)) / np.sqrt(K)).astype(np.float32)
    Phi = torch.tensor(P0, device="cuda")
    t.cp_step(lib.DeviceCSR.from_corpus(c), Phi, 0.0, want_loss=loss)  # what a step before leaves (rows of Q)
    bad = c.indptr.copy()
    bad[0] = -1
    try:
        t.cp_step(lib.DeviceCSR.from_arrays(bad, c.indices, c.counts, V), Phi, 1e-3, want_loss=loss)
        t.sync()
        raise AssertionError("a negative offset was accepted")
    except lib.TLDAError:
        pass
    assert np.array_equal(Phi.cpu().numpy(), P0)
    # a valid batch of the same words, whose sums nothing may be left in
    grad = torch.empty_like(Phi)
    t.cp_step(lib.DeviceCSR.from_corpus(c), Phi, 0.0, grad=grad, want_loss=loss)
    t.sync()
    g = O.cp_grad_implicit(c.indptr, c.indices, c.counts, V, W, m1, P0.astype(np.float64), 1.5, 0.0)
    assert C.rel(grad.cpu().numpy(), g["grad"]) < tol
    t.close()
