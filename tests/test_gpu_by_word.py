"""The FP32 step without the loss (data term regrouped by word) at the edges of its
tiles, staged rows and copies, against the FP64 oracle; and the touched words found
one batch ahead in a pass."""
import numpy as np
import pytest
import torch

import tlda_synth as ts
from oracle import tlda_oracle as O

from . import _cases as C

pytestmark = pytest.mark.gpu


def _corpus(rng, V, lens, hot):
    """Documents of the given numbers of words; word 0 in a share `hot` of them."""
    rows, idx, cnt = [0], [], []
    for n in lens:
        w = rng.choice(V - 1, size=n, replace=False) + 1 if n else np.zeros(0, dtype=np.int64)
        if n and rng.random() < hot:
            w[0] = 0
        idx += list(np.sort(w))
        cnt += list(rng.integers(1, 4, size=n))
        rows.append(len(idx))
    return ts.Corpus(np.array(rows, dtype=np.int64), np.array(idx, dtype=np.int32), np.array(cnt, dtype=np.int32), None, V)


def _model(lib, rng, V, K, D, **kw):
    W = rng.standard_normal((V, D)).astype(np.float32)
    m1 = (W.mean(axis=0) + 0.1 * rng.standard_normal(D)).astype(np.float32)
    t = lib.TLDA(V, K, dim=D, alpha0=1.5, max_batch=512, **kw)
    t.set_whitening(torch.tensor(W), torch.tensor(m1))
    return t, W.astype(np.float64), m1.astype(np.float64)


# topics and features below, at and above 64 and 128 and of every remainder by 4;
# documents of every length to 40 words (rows staged at once, 32-word chunks) and of 70 and 130
@pytest.mark.parametrize("K,D", [(1, 1), (3, 5), (10, 10), (63, 64), (64, 64), (50, 100), (65, 66), (100, 100), (128, 128),
                                 (64, 129), (129, 130), (200, 200), (300, 301)])
@pytest.mark.parametrize("same", [True, False])
def test_step_by_word(lib, K, D, same):
    rng = np.random.default_rng(K + 1000 * D)
    V = 1000
    c = _corpus(rng, V, list(range(41)) + [70, 130] * 2 + list(rng.integers(3, 20, 150)), 0.8)
    t, W, m1 = _model(lib, rng, V, K, D, same_token=same)
    P0 = (rng.standard_normal((D, K)) / np.sqrt(D)).astype(np.float32)
    Phi = torch.tensor(P0, device="cuda")
    grad = torch.empty_like(Phi)
    dev = lib.DeviceCSR.from_corpus(c)
    for _ in range(2):  # the second step starts from what the first one left behind
        Phi.copy_(torch.tensor(P0))
        t.cp_step(dev, Phi, 1e-3, grad=grad)
    t.sync()
    g = O.cp_grad_implicit(c.indptr, c.indices, c.counts, V, W, m1, P0.astype(np.float64), 1.5, 0.0, same_token=same)
    # FP32 rounding of sums of some thousand terms: the bar of the FP32 form
    assert C.rel(grad.cpu().numpy(), g["grad"]) < 1e-5
    assert C.rel(Phi.cpu().numpy(), P0 - 1e-3 * g["grad"]) < 1e-5
    t.close()


@pytest.mark.parametrize("precision,K", [("fp32", 40), ("fp32", 100), ("bf16", 40), ("bf16", 150)])
def test_pass_finds_words_ahead(lib, precision, K):
    """Batches of very different size, empty ones among them, a word in most documents: the device-input pass
    (words found a batch ahead) steps as the host-input pass and as single steps do."""
    rng = np.random.default_rng(K)
    V = 700
    c = _corpus(rng, V, list(rng.integers(0, 25, 900)), 0.9)
    offs = [0, 1, 1, 300, 310, 310, 822, 900]
    t, _, _ = _model(lib, rng, V, K, K, precision=precision)
    P0 = torch.tensor((rng.standard_normal((K, K)) / np.sqrt(K)).astype(np.float32), device="cuda")
    dev = lib.DeviceCSR.from_corpus(c)
    out = []
    for kind in ("device", "device", "host", "steps"):
        Phi = P0.clone()
        if kind == "steps":
            for a, b in zip(offs, offs[1:]):
                t.cp_step(lib.DeviceCSR(dev.indptr[a:b + 1], dev.indices, dev.counts, V), Phi, 1e-5)
        else:
            src = lib.DeviceCSR.from_corpus(c, device="cpu", pin=True) if kind == "host" else dev
            t.cp_pass(src, offs, Phi, 1e-5, host_input=kind == "host")
        t.sync()
        out.append(Phi.cpu().numpy().astype(np.float64))
    upd = np.abs(out[0] - P0.cpu().numpy()).max()
    assert upd > 0
    for o in out[1:]:  # the order of the FP32 adds, and BF16 roundings that flip with it
        assert np.abs(o - out[0]).max() < (1e-4 if precision == "fp32" else 1e-2) * upd
    t.close()


def test_corrupt_batch_leaves_no_trace(lib):
    """After a batch whose offsets decrease at the end (words outside the batch's range), a valid step is right."""
    rng = np.random.default_rng(3)
    V, K = 500, 30
    c = _corpus(rng, V, list(rng.integers(3, 20, 200)), 0.5)
    t, W, m1 = _model(lib, rng, V, K, K)
    P0 = (rng.standard_normal((K, K)) / np.sqrt(K)).astype(np.float32)
    Phi = torch.tensor(P0, device="cuda")
    bad = c.indptr.copy()
    bad[-1] = bad[-3]
    dev_bad = lib.DeviceCSR.from_arrays(bad, c.indices, c.counts, V)
    t.cp_step(dev_bad, Phi, 1e-3)
    with pytest.raises(lib.TLDAError):
        t.sync()
    assert np.array_equal(Phi.cpu().numpy(), P0)
    grad = torch.empty_like(Phi)
    t.cp_step(lib.DeviceCSR.from_corpus(c), Phi, 0.0, grad=grad)
    t.sync()
    g = O.cp_grad_implicit(c.indptr, c.indices, c.counts, V, W, m1, P0.astype(np.float64), 1.5, 0.0)
    assert C.rel(grad.cpu().numpy(), g["grad"]) < 1e-5
    t.close()
