"""Passes that return their losses: device input, host input and single steps agree."""
import numpy as np
import pytest
import torch

from .test_gpu_by_word import _corpus, _model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("same", [True, False])
@pytest.mark.parametrize("precision,K", [("fp32", 40), ("fp32", 150), ("bf16", 40), ("bf16", 150)])
def test_losses_of_a_pass(lib, precision, K, same):
    rng = np.random.default_rng(K)
    V = 700
    c = _corpus(rng, V, list(rng.integers(3, 25, 900)), 0.9)
    offs = [0, 1, 1, 300, 310, 310, 822, 900]  # batches of very different size, empty ones among them
    t, _, _ = _model(lib, rng, V, K, K, precision=precision, same_token=same)
    P0 = torch.tensor((rng.standard_normal((K, K)) / np.sqrt(K)).astype(np.float32), device="cuda")
    dev, host = lib.DeviceCSR.from_corpus(c), lib.DeviceCSR.from_corpus(c, device="cpu", pin=True)
    out = []
    for kind in ("steps", "device", "host", "device"):
        Phi = P0.clone()
        if kind == "steps":
            loss = [t.cp_step(lib.DeviceCSR(dev.indptr[a:b + 1], dev.indices, dev.counts, V), Phi, 1e-5, want_loss=True)
                    for a, b in zip(offs, offs[1:])]
        else:
            loss = t.cp_pass(host if kind == "host" else dev, offs, Phi, 1e-5, host_input=kind == "host", losses=True)
        t.sync()
        out.append((np.array(loss), Phi.cpu().numpy().astype(np.float64)))
    t.close()
    (l0, P), tol = out[0], 1e-4 if precision == "fp32" else 1e-2
    upd = np.abs(P - P0.cpu().numpy()).max()
    assert upd > 0 and (l0[[1, 4]] == 0).all()
    for l, Q in out[1:]:  # the order of the FP32 adds, and BF16 roundings that flip with it
        assert np.abs(Q - P).max() <= tol * upd
        assert np.abs(l - l0).max() <= tol * np.abs(l0).max()
