"""Document-topic VI at the edges of its topic groups (32 topics a lane slot) and
word groups (four words at a time, some kept in registers), against the oracle."""
import numpy as np
import pytest

import tlda_synth as ts
from oracle import tlda_oracle as O

from . import _cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 31, 32, 33, 64, 65, 96, 97, 128, 129, 192, 193, 256, 257, 384, 385, 512])
def test_doc_topics_at_group_edges(lib, K):
    rng = np.random.default_rng(K)
    V = 300
    mu = rng.dirichlet(np.full(V, 0.1), size=K).T.astype(np.float32).astype(np.float64)
    mu[rng.integers(0, V, 5)] = 0.0  # words no topic uses
    alpha = rng.uniform(0.005, 0.5, size=K).astype(np.float32).astype(np.float64)
    # every document length from 0 to 40 words, and longer ones than any group kept in registers
    lens = list(range(41)) + [63, 64, 65, 130]
    rows, idx, cnt = [0], [], []
    for n in lens:
        idx += list(np.sort(rng.choice(V, size=n, replace=False)))
        cnt += list(rng.integers(1, 5, size=n))
        rows.append(len(idx))
    c = ts.Corpus(np.array(rows, dtype=np.int64), np.array(idx, dtype=np.int32), np.array(cnt, dtype=np.int32), None, V)
    dev = lib.DeviceCSR.from_arrays(c.indptr, c.indices, c.counts, V)
    theta, gamma = lib.doc_topics(dev, mu, alpha, 8, want_gamma=True)
    th_o, ga_o = O.doc_topics(c.indptr, c.indices, c.counts, V, mu, alpha, 8)
    # FP32 rounding of exp(digamma) (some 10 units of 2^-24 for exponents below 16, more below) over 8 rounds
    assert C.rel(theta.cpu().numpy(), th_o) < 1e-5
    assert C.rel(gamma.cpu().numpy(), ga_o) < 1e-5
