"""The allocation-free CP step above 128 features, where the data term is folded,
multiplied and cleared by kernels of their own, against the context step."""
import numpy as np
import pytest
import torch

from tests import _cases as C
from tests.test_gpu_by_word import _corpus
from tests.test_zz_no_alloc import TOL32, _noalloc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,D,K", [(500, 130, 130), (1000, 200, 50), (400, 129, 65)])
def test_noalloc_above_128_features(lib, V, D, K):
    rng = np.random.default_rng(D)
    W = rng.standard_normal((V, D)).astype(np.float32)
    m1 = W.mean(axis=0).astype(np.float32)
    ctx = lib.TLDA(V, K, dim=D, alpha0=1.5, max_batch=512)
    ctx.set_whitening(torch.tensor(W), torch.tensor(m1))
    P0 = torch.tensor((rng.standard_normal((D, K)) / np.sqrt(D)).astype(np.float32), device="cuda")
    Wd, m1d = torch.tensor(W, device="cuda"), torch.tensor(m1, device="cuda")
    g, g_ref = torch.empty_like(P0), torch.empty_like(P0)
    err = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    for n in (200, 60, 200):  # each batch on what the one before left
        b = lib.DeviceCSR.from_corpus(_corpus(rng, V, list(rng.integers(0, 25, n)), 0.7))
        Phi, ref = P0.clone(), P0.clone()
        ctx.cp_step(b, ref, 1e-3, grad=g_ref)
        ctx.sync()
        assert _noalloc(lib, b, Wd, m1d, D, K, 1.5, 0.0, Phi, 1e-3, g, err) == lib.OK
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        assert C.rel(g.cpu().numpy(), g_ref.cpu().numpy()) < TOL32
        assert C.rel(Phi.cpu().numpy(), ref.cpu().numpy()) < TOL32
    ctx.close()
