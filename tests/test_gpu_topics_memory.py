"""Topics read on the host leave no large buffer behind on the device."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,K", [(30000, 100), (60000, 100)])  # 24 MB, which a context may keep, and 48 MB
def test_memory_after_topics(lib, V, K):
    rng = np.random.default_rng(0)
    W = torch.tensor(rng.standard_normal((V, K)).astype(np.float32))
    Phi = torch.tensor(rng.standard_normal((K, K)).astype(np.float32), device="cuda")
    small = lib.TLDA(200, 4, max_batch=64)  # the kernels are loaded
    small.set_whitening(torch.tensor(rng.standard_normal((200, 4)).astype(np.float32)), torch.zeros(4))
    small.unwhiten_topics(torch.eye(4, device="cuda"))
    t = lib.TLDA(V, K, max_batch=64)
    t.set_whitening(W, torch.zeros(K))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    mu, _ = t.unwhiten_topics(Phi)
    torch.cuda.synchronize()
    # the small workspace (some D x D and V words), in the allocator's 2 MB pages
    assert before - torch.cuda.mem_get_info()[0] <= (40 << 20)
    again, _ = t.unwhiten_topics(Phi)
    assert np.abs(again - mu).max() <= 1e-12 and np.abs(mu.sum(axis=0) - 1.0).max() <= 1e-9
    t.close()
    small.close()
