"""What the library's speed is measured on: the calls that make up an online Tensor LDA job.

A job runs, in order: the moments and the whitening of a corpus (`fit`) or their one-pass sketch
(`sketch`, `online`), minibatch passes of CP steps over documents on the device or in host memory
(`pass`), single steps as a differentiable loss (`loss`), whitened batches (`whiten`), and at the end the
topics (`topics`) and the documents' topic proportions (`vi`).  The sizes are those of the seeded
workloads of this repository (500 to 100,000 words, 2 to 300 topics, minibatches of 512 to 65,536
documents); the corpora are drawn here, from the model of latent Dirichlet allocation.
"""
import math
import random

import numpy as np
import torch

from paper_2511_07809_gb300 import tlda

GPU = "cuda"

# One corpus shape per workload: vocabulary, topics, alpha0, mean document length, topic prior
# (concentration per word; zipf: exponent of its shape, over one word order or one per topic).
SMALL = {"V": 500, "K": 10, "alpha0": 1.0, "length": 50, "beta": 0.1, "zipf": 0.0, "own_order": False}
TWEET = {"V": 5000, "K": 50, "alpha0": 1.0, "length": 30, "beta": 0.05, "zipf": 1.1, "own_order": False}
STREAM = {"V": 20000, "K": 100, "alpha0": 2.0, "length": 12, "beta": 0.1, "zipf": 0.0, "own_order": False}
BILLION = {"V": 100000, "K": 300, "alpha0": 5.0, "length": 15, "beta": 0.05, "zipf": 1.07, "own_order": True}

LR = {"small": 1e-2, "stream": 2e-3, "tweet": 2e-4, "wide": 1e-4}


def listed():
    return [
        # one step of a small topic model as a loss with its gradient, as a user's optimiser calls it
        {"name": "loss_small", "kind": "loss", "prec": "fp32", "docs": 1000, **SMALL},
        # the streaming pass over uneven minibatches, corpus on the device: the headline
        {"name": "pass_stream_bf16", "kind": "pass", "prec": "bf16", "lo": 512, "hi": 8192, "batches": 64,
         "host": False, "lr": LR["stream"], **STREAM},
        # the same from pinned host memory, every step's loss read back
        {"name": "pass_stream_host", "kind": "pass", "prec": "bf16", "lo": 512, "hi": 8192, "batches": 160,
         "host": True, "lr": LR["stream"], **STREAM},
        # the same in the plain FP32 form
        {"name": "pass_stream_fp32", "kind": "pass", "prec": "fp32", "lo": 512, "hi": 8192, "batches": 24,
         "host": False, "lr": LR["stream"], **STREAM},
        # minibatches of tweets: half the topics, longer documents, a shared Zipf head
        {"name": "pass_tweet_bf16", "kind": "pass", "prec": "bf16", "lo": 4096, "hi": 4096, "batches": 24,
         "host": False, "lr": LR["tweet"], **TWEET},
        # the widest model: 100,000 words, 300 topics, large minibatches
        {"name": "pass_billion_bf16", "kind": "pass", "prec": "bf16", "lo": 65536, "hi": 65536, "batches": 4,
         "host": False, "lr": LR["wide"], **BILLION},
        # the whitened batch alone (the SpMM of the path)
        {"name": "whiten_stream", "kind": "whiten", "prec": "fp32", "docs": 8192, **STREAM},
        # exact moments of a corpus in chunks, and the whitening from their eigenpairs
        {"name": "fit_tweet", "kind": "fit", "prec": "fp32", "docs": 200000, "chunks": 4, **TWEET},
        # a block of the fully online mode after a resume: sketch, whitening rebuilt, factors carried, CP steps
        {"name": "online_stream", "kind": "online", "prec": "bf16", "r": 216, "seen": 200000, "lo": 512,
         "hi": 8192, "batches": 64, "lr": 5e-4, **STREAM},
        # the one-pass sketch of a large chunk of documents
        {"name": "sketch_billion", "kind": "sketch", "prec": "bf16", "r": 512, "docs": 300000, **BILLION},
        # the topics of a finished model, read on the host
        {"name": "topics_stream", "kind": "topics", "prec": "fp32", **STREAM},
        # topic proportions of documents under finished topics
        {"name": "vi_stream", "kind": "vi", "iters": 20, "docs": 300000, **STREAM},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["loss", "pass", "pass", "pass", "whiten", "fit", "online", "sketch", "topics", "vi"])
    prec = rng.choice(["fp32", "bf16"])
    zipf = rng.choice([0.0, 1.1])

    def model(V, K, length):
        # a shared Zipf head leaves many topics no second moment of full rank: one order per topic above 64
        return {"V": V, "K": K, "alpha0": rng.choice([1.0, 2.0] if kind in ("fit", "online") else [1.0, 2.0, 5.0]), "length": length,
                "beta": 0.1 if zipf == 0.0 else 0.05, "zipf": zipf, "own_order": zipf > 0 and (K > 64 or rng.random() < 0.5)}

    if kind == "loss":
        V = _log(rng, 500, 20000)
        return {"kind": kind, "prec": prec, "docs": _log(rng, 64, 8192), **model(V, _log(rng, 2, min(200, V // 10)), _log(rng, 12, 50))}
    if kind == "pass":
        shape = rng.choice(["narrow", "stream", "wide"])
        host = rng.random() < 0.3
        if shape == "narrow":
            hi = _log(rng, 512, 8192)
            m = model(_log(rng, 700, 20000), _log(rng, 5, 64), _log(rng, 12, 50))
        elif shape == "stream":
            hi = _log(rng, 1024, 8192)
            m = model(_log(rng, 5000, 30000), rng.randint(65, 128), _log(rng, 8, 30))
        else:
            hi = _log(rng, 4096, 50000)
            m = model(_log(rng, 20000, 100000), rng.randint(129, 300), _log(rng, 10, 20))
        return {"kind": kind, "prec": prec, "lo": max(1, hi // rng.choice([1, 2, 16])), "hi": hi,
                "batches": min(200, max(3, 400000 // hi)) if shape != "wide" else 4, "host": host, "lr": 1e-4, **m}
    if kind == "whiten":
        return {"kind": kind, "prec": "fp32", "docs": _log(rng, 200, 30000), **model(_log(rng, 3000, 50000), _log(rng, 10, 300), _log(rng, 10, 50))}
    if kind == "fit":
        return {"kind": kind, "prec": prec, "docs": _log(rng, 100000, 200000), "chunks": rng.randint(1, 5),
                **model(_log(rng, 500, 5000), rng.randint(5, 50), _log(rng, 25, 40))}
    if kind == "online":
        K = rng.randint(20, 100)
        m = model(_log(rng, 2000, 20000), K, _log(rng, 20, 40))
        return {"kind": kind, "prec": prec, "r": 2 * K + 2 * rng.randint(4, 14), "seen": _log(rng, 200000, 300000), "lo": 512, "hi": 4096,
                "batches": rng.randint(8, 64), "lr": 1e-4, **m}
    if kind == "sketch":
        K = rng.randint(50, 200)
        return {"kind": kind, "prec": prec, "r": 2 * rng.randint(K // 2 + 8, 256), "docs": _log(rng, 20000, 300000), **model(_log(rng, 5000, 100000), K, _log(rng, 10, 20))}
    if kind == "topics":
        return {"kind": kind, "prec": prec, **model(_log(rng, 1000, 30000), _log(rng, 10, 100), 12)}
    return {"kind": kind, "iters": rng.choice([10, 20, 30]), "docs": _log(rng, 5000, 200000), **model(_log(rng, 2000, 20000), _log(rng, 10, 200), _log(rng, 10, 50))}


# ------------------------------------------------------------------ inputs
def _gen(seed, what):
    g = torch.Generator(device=GPU)
    g.manual_seed((int(seed) * 1000003 + what) % (1 << 62))
    return g


def _topics(c, seed):
    """mu (V x K float64, columns sum to 1) and the integer tables that words are drawn from."""
    V, K = c["V"], c["K"]
    g = _gen(seed, 1)
    conc = torch.full((K, V), c["beta"], dtype=torch.float64, device=GPU)
    if c["zipf"] > 0:
        p = torch.arange(1, V + 1, dtype=torch.float64, device=GPU) ** -c["zipf"]
        p = p * (c["beta"] * V / p.sum())
        if c["own_order"]:
            order = torch.rand((K, V), generator=g, device=GPU).argsort(dim=1)
            conc = p[order]
        else:
            conc = p.expand(K, V).contiguous()
    w = torch._standard_gamma(conc, generator=g)
    return _tables(w / w.sum(dim=1, keepdim=True))


def _tables(p):
    """Rows of probabilities as whole numbers: (p as rounded, its running sums over all rows, first sums, totals)."""
    n = (p * 2.0 ** 30).to(torch.int64)
    cum = n.reshape(-1).cumsum(0)
    total = n.sum(dim=1)
    return n, cum, total.cumsum(0) - total, total


def _pick(tables, rows, g):
    """One column of each given row, drawn by its probabilities."""
    n, cum, first, total = tables
    u = torch.rand(rows.numel(), generator=g, device=GPU, dtype=torch.float64)
    key = first[rows] + torch.minimum((u * total[rows]).to(torch.int64), total[rows] - 1)
    return torch.searchsorted(cum, key, right=True) % n.shape[1]


def _corpus(c, seed, docs, tables, stream=0):
    """`docs` documents of the model as CSR arrays (int32, GPU)."""
    V, K = c["V"], c["K"]
    g = _gen(seed, 1000 + stream)
    lens = torch.poisson(torch.full((docs,), float(c["length"]), device=GPU), generator=g).to(torch.int64).clamp_(min=3)
    theta = torch._standard_gamma(torch.full((docs, K), c["alpha0"] / K, device=GPU), generator=g).double()
    theta = _tables((theta + 1e-30) / (theta + 1e-30).sum(dim=1, keepdim=True))
    doc = torch.repeat_interleave(torch.arange(docs, device=GPU), lens)
    word = _pick(tables, _pick(theta, doc, g), g)
    key, counts = torch.unique_consecutive((doc * V + word).sort().values, return_counts=True)
    per = torch.bincount(key // V, minlength=docs)
    indptr = torch.zeros(docs + 1, dtype=torch.int32, device=GPU)
    indptr[1:] = per.cumsum(0).to(torch.int32)
    return indptr, (key % V).to(torch.int32), counts.to(torch.int32)


def _mu(tables):
    n = tables[0].double()
    return (n / n.sum(dim=1, keepdim=True)).t().contiguous()


def _whitening(mu):
    """W and m1 (float32) of the model's own second moment, the mean of mu_k mu_k^T over the topics."""
    K = mu.shape[1]
    lam, E = torch.linalg.eigh(mu.t() @ mu / K)
    W = (mu @ E).flip(1) / (lam.flip(0) * math.sqrt(K))
    return W.float().contiguous(), (W.t() @ mu.mean(dim=1)).float().contiguous()


def _phi(K, seed):
    return torch.randn((K, K), generator=_gen(seed, 2), device=GPU) / math.sqrt(K)


def _offsets(c, seed):
    rng = random.Random(int(seed) * 7919 + 5)
    off = [0]
    for _ in range(c["batches"]):
        off.append(off[-1] + rng.randint(c["lo"], c["hi"]))
    return np.asarray(off, dtype=np.int64)


def _signs(V, r, seed):
    return torch.randint(0, 2, (V, r), generator=_gen(seed, 3), device=GPU).double() * 2 - 1


def _csr(c, arrays, host=False):
    a = [x.cpu().pin_memory() for x in arrays] if host else list(arrays)
    return tlda.DeviceCSR(a[0], a[1], a[2], c["V"])


def _inputs(c, seed):
    """Everything the call reads, as tensors."""
    kind, K = c["kind"], c["K"]
    tables = _topics(c, seed)
    mu = _mu(tables)
    d = {"mu": mu}
    if kind in ("loss", "pass", "whiten", "online", "topics"):
        d["W"], d["m1"] = _whitening(mu)
    if kind in ("loss", "pass", "online"):
        d["Phi"] = _phi(K, seed)
    if kind in ("pass", "online"):
        d["off"] = _offsets(c, seed)
        d["csr"] = _corpus(c, seed, int(d["off"][-1]), tables)
    if kind in ("loss", "whiten", "sketch", "vi"):
        d["csr"] = _corpus(c, seed, c["docs"], tables)
    if kind == "fit":
        cut = [c["docs"] * i // c["chunks"] for i in range(c["chunks"] + 1)]
        d["chunks"] = [_corpus(c, seed, b - a, tables, stream=a) for a, b in zip(cut, cut[1:])]
    if kind in ("online", "sketch"):
        d["Omega"] = _signs(c["V"], c["r"], seed)
    if kind == "online":
        # the sketch and the counts that a checkpoint after `seen` documents holds
        d["Z"], d["C"], d["TS"] = _sketch(_corpus(c, seed, c["seen"], tables, stream=1), d["Omega"])
    if kind == "topics":
        # factors near the decomposition, as a pass leaves them
        v = d["W"].t() @ mu.float() / math.sqrt(K)
        d["Phi"] = ((v + 0.02 * torch.randn(v.shape, generator=_gen(seed, 4), device=GPU) * v.std()) * K ** (1 / 6)).contiguous()
    if kind == "vi":
        d["mu32"] = mu.float().contiguous()
        d["alpha"] = torch.full((K,), c["alpha0"] / K, device=GPU)
    return d


def prepare(case, seed):
    c = case
    d = _inputs(c, seed)
    s = {"case": c, "d": d}
    kind = c["kind"]
    if kind == "vi":
        s["csr"] = _csr(c, d["csr"])
        return s
    most = c.get("hi") or c.get("docs") or 1024
    s["t"] = t = tlda.TLDA(c["V"], c["K"], alpha0=c["alpha0"], precision=c["prec"], max_batch=min(most, 65536) if kind not in ("fit", "sketch") else 1024)
    if "W" in d:
        t.set_whitening(d["W"], d["m1"])
    if "csr" in d:
        s["csr"] = _csr(c, d["csr"], c.get("host", False))
    if "chunks" in d:
        s["chunks"] = [_csr(c, a) for a in d["chunks"]]
    if "Phi" in d:
        s["Phi"] = d["Phi"].clone()
    if kind == "loss":
        s["Phi"].requires_grad_(True)
    if kind == "whiten":
        s["X"] = torch.empty((c["docs"], c["K"]), device=GPU)
    if kind in ("online", "sketch"):
        t.online_begin(d["Omega"])
    if kind in ("pass", "online") and c["prec"] == "bf16" and 64 < c["K"] <= 128:
        t.autotune(fixed=18)  # one tile size, so that two runs add in the same order
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    c, d, t = s["case"], s["d"], s.get("t")
    kind = c["kind"]
    if kind == "loss":
        s["Phi"].grad = None
        loss = tlda.tlda_loss(s["Phi"], t, s["csr"])
        loss.backward()
        return {"loss": loss.detach(), "grad": s["Phi"].grad}
    if kind == "pass":
        s["Phi"].copy_(d["Phi"])
        losses = t.cp_pass(s["csr"], d["off"], s["Phi"], c["lr"], host_input=c["host"], losses=c["host"])
        return {"Phi": s["Phi"], "losses": losses} if c["host"] else {"Phi": s["Phi"]}
    if kind == "whiten":
        return t.whiten_batch(s["csr"], s["X"])
    if kind == "fit":
        t.fit(s["chunks"])
        W, m1, ev = t.get_whitening()
        C, T, S2, S3 = t.get_counts()
        return {"W": W, "m1": m1, "ev": ev, "C": C, "T": T, "S2": S2, "S3": S3}
    if kind == "online":
        t.set_whitening(d["W"], d["m1"])
        t.online_set_sketch(d["Z"], d["C"], d["TS"])
        s["Phi"].copy_(d["Phi"])
        losses = t.online_pass(s["csr"], d["off"], s["Phi"], c["lr"], rewhiten_every=c["batches"], losses=True)
        W, m1, ev = t.get_whitening()
        return {"Phi": s["Phi"], "losses": losses, "W": W, "m1": m1, "ev": ev}
    if kind == "sketch":
        t.online_begin(d["Omega"])
        t.online_accumulate(s["csr"])
        Z, C, TS = t.online_sketch()
        return {"Z": Z, "C": C, "TS": TS}
    if kind == "topics":
        mu, alpha = t.unwhiten_topics(s["Phi"])
        return {"mu": mu, "alpha": alpha}
    theta, gamma = tlda.doc_topics(s["csr"], d["mu32"], d["alpha"], n_iter=c["iters"], want_gamma=True)
    return {"theta": theta, "gamma": gamma}


def work(case):
    c, kind = case, case["kind"]
    V, K, L = c["V"], c["K"], c["length"]

    def step(B):
        """Bytes and operations of one CP step over B documents: the CSR once, the factors in and out; Q = U Phi
        and U^T B over the words met, the sums over the nonzeros, the terms of the factors alone."""
        nnz, met = 0.95 * B * L, min(V, 0.95 * B * L)
        return 8 * nnz + 4 * B, 4 * met * K * K + 11 * nnz * K + 4 * K ** 3

    table = (2 if c.get("prec") == "bf16" else 4) * V * K
    if kind == "loss":
        b, f = step(c["docs"])
        return {"bytes": b + min(table, table / V * 0.95 * c["docs"] * L) + 8 * K * K, "flops": f}
    if kind == "pass":
        b, f = step((c["lo"] + c["hi"]) / 2)
        return {"bytes": b * c["batches"] + table + 8 * K * K, "flops": f * c["batches"]}
    if kind == "whiten":
        nnz = 0.95 * c["docs"] * L
        return {"bytes": 8 * nnz + 4 * c["docs"] + table + 4 * c["docs"] * K, "flops": 2 * nnz * K}
    if kind == "fit":
        # one product of the second moment with K vectors and its eigenproblem in that space, at the least
        nnz = 0.95 * c["docs"] * L
        return {"bytes": 8 * nnz + 4 * c["docs"] + 8 * V * V + 4 * V * K + 8 * V,
                "flops": nnz * 0.95 * L + 2 * V * V * K + 4 * V * K * K + 9 * K ** 3}
    if kind == "online":
        B, r = c["batches"] * (c["lo"] + c["hi"]) / 2, c["r"]
        b, f = step((c["lo"] + c["hi"]) / 2)
        nnz = 0.95 * B * L
        return {"bytes": b * c["batches"] + 24 * V * r + 8 * V * K, "flops": f * c["batches"] + 5 * nnz * r + 6 * V * r * r + 9 * r ** 3 + 4 * V * K * K}
    if kind == "sketch":
        nnz, r = 0.95 * c["docs"] * L, c["r"]
        return {"bytes": 8 * nnz + 4 * c["docs"] + 16 * V * r + 8 * V, "flops": 5 * nnz * r}
    if kind == "topics":
        return {"bytes": 4 * V * K + 8 * V * K, "flops": 4 * V * K * K + 3 * K ** 3}
    nnz = 0.95 * c["docs"] * L
    return {"bytes": 8 * nnz + 4 * c["docs"] + 4 * V * K + 8 * c["docs"] * K, "flops": c["iters"] * (5 * nnz * K + 20 * c["docs"] * K)}


# ------------------------------------------------------------------ the same in 64 bits
def _rows(csr):
    indptr, indices, counts = csr
    lens = (indptr[1:] - indptr[:-1]).long()
    return torch.repeat_interleave(torch.arange(lens.numel(), device=GPU), lens), indices.long(), counts.double()


def _sketch(csr, Omega):
    """Z = (F^T F - diag(F^T 1)) Omega, the word counts and the sums of L, L(L-1), L(L-1)(L-2)."""
    doc, word, f = _rows(csr)
    V, docs = Omega.shape[0], csr[0].numel() - 1
    L = torch.zeros(docs, dtype=torch.float64, device=GPU).index_add_(0, doc, f)
    C = torch.zeros(V, dtype=torch.float64, device=GPU).index_add_(0, word, f)
    Z = -C[:, None] * Omega
    block = max(1, 1 << 28 >> 9)  # documents' sums in pieces, by nonzeros
    edges = torch.searchsorted(csr[0].long(), torch.arange(0, word.numel() + block, block, device=GPU)).clamp_(max=docs).tolist()
    edges = sorted(set([0] + edges + [docs]))
    for a, b in zip(edges, edges[1:]):
        lo, hi = int(csr[0][a]), int(csr[0][b])
        if hi > lo:
            S = torch.zeros((b - a, Omega.shape[1]), dtype=torch.float64, device=GPU).index_add_(0, doc[lo:hi] - a, f[lo:hi, None] * Omega[word[lo:hi]])
            Z.index_add_(0, word[lo:hi], f[lo:hi, None] * S[doc[lo:hi] - a])
    TS = torch.stack([L.sum(), (L * (L - 1)).sum(), (L * (L - 1) * (L - 2)).sum()])
    return Z, C.round().long(), TS.round().long()


def _step64(csr, d0, d1, W, m1, Phi, alpha0):
    """Loss and gradient of one CP step (theta = 0) over documents [d0, d1)."""
    lo, hi = int(csr[0][d0]), int(csr[0][d1])
    doc, word, f = _rows((csr[0][d0:d1 + 1], csr[1][lo:hi], csr[2][lo:hi]))
    K = Phi.shape[1]
    L = torch.zeros(d1 - d0, dtype=torch.float64, device=GPU).index_add_(0, doc, f)
    S3 = float((L * (L - 1) * (L - 2)).sum())
    uw, at = torch.unique(word, return_inverse=True)
    U = W[uw] - m1
    q = (U @ Phi)[at]
    y = torch.zeros((d1 - d0, K), dtype=torch.float64, device=GPU).index_add_(0, doc, f[:, None] * q)
    r = torch.zeros_like(y).index_add_(0, doc, f[:, None] * q * q)
    b = f[:, None] * ((y * y - r)[doc] + 2 * q * q - 2 * q * y[doc])
    G12 = U.t() @ torch.zeros((uw.numel(), K), dtype=torch.float64, device=GPU).index_add_(0, at, b)
    a, n2, gram = m1 @ Phi, (Phi * Phi).sum(dim=0), Phi.t() @ Phi
    G3 = 2 * Phi * a + m1[:, None] * n2 - 2 * m1[:, None] * a * a
    scale = (alpha0 + 1) * (alpha0 + 2) / 2 / S3 if S3 else 0.0
    data = (y ** 3 - 3 * y * r).sum() + 2 * (f[:, None] * q ** 3).sum()
    if not S3:
        return torch.zeros((), dtype=torch.float64, device=GPU), torch.zeros_like(Phi)
    loss = 0.5 * (gram ** 3).sum() - (3 * a * n2 - 2 * a ** 3).sum() - scale * data
    return loss, 3 * Phi @ (gram * gram) - 3 * (scale * G12 + G3)


def _pass64(c, d, W, m1, Phi):
    losses = []
    for a, b in zip(d["off"], d["off"][1:]):
        loss, grad = _step64(d["csr"], int(a), int(b), W, m1, Phi, c["alpha0"])
        losses.append(loss)
        Phi = Phi - c["lr"] * grad
    return Phi, torch.stack(losses)


def _signed(U):
    """Each column's entry of largest magnitude made positive."""
    top = U.gather(0, U.abs().argmax(dim=0, keepdim=True))
    return U * torch.where(top < 0, -1.0, 1.0)


def exact(case, seed):
    c = case
    d = _inputs(c, seed)
    kind, K, V = c["kind"], c["K"], c["V"]
    if kind == "loss":
        loss, grad = _step64(d["csr"], 0, c["docs"], d["W"].double(), d["m1"].double(), d["Phi"].double(), c["alpha0"])
        return {"loss": loss, "grad": grad}
    if kind == "pass":
        Phi, losses = _pass64(c, d, d["W"].double(), d["m1"].double(), d["Phi"].double())
        return {"Phi": Phi, "losses": losses} if c["host"] else {"Phi": Phi}
    if kind == "whiten":
        doc, word, f = _rows(d["csr"])
        return torch.zeros((c["docs"], K), dtype=torch.float64, device=GPU).index_add_(0, doc, f[:, None] * (d["W"].double() - d["m1"].double())[word])
    if kind == "fit":
        if V > 6000:
            return None
        P = torch.zeros((V, V), dtype=torch.float64, device=GPU)
        C, TS = torch.zeros(V, dtype=torch.float64, device=GPU), torch.zeros(3, dtype=torch.float64, device=GPU)
        for csr in d["chunks"]:
            doc, word, f = _rows(csr)
            docs = csr[0].numel() - 1
            C.index_add_(0, word, f)
            L = torch.zeros(docs, dtype=torch.float64, device=GPU).index_add_(0, doc, f)
            TS += torch.stack([L.sum(), (L * (L - 1)).sum(), (L * (L - 1) * (L - 2)).sum()])
            for a in range(0, docs, 20000):  # sums of whole numbers far below 2^24: exact in 32 bits
                b = min(docs, a + 20000)
                lo, hi = int(csr[0][a]), int(csr[0][b])
                F = torch.zeros((b - a, V), device=GPU)
                F[doc[lo:hi] - a, word[lo:hi]] = f[lo:hi].float()
                P += (F.t() @ F).double()
        P -= torch.diag(C)
        M1 = C / TS[0]
        lam, E = torch.linalg.eigh((c["alpha0"] + 1) / TS[1] * P - c["alpha0"] * torch.outer(M1, M1))
        ev = lam[-K:].flip(0)
        W = _signed(E[:, -K:].flip(1)) / ev.sqrt()
        return {"W": W, "m1": W.t() @ M1, "ev": ev, "C": None, "T": None, "S2": None, "S3": None}
    if kind == "online":
        Z, C, TS = _sketch(d["csr"], d["Omega"])
        Z, C, TS = Z + d["Z"], C + d["C"], TS + d["TS"]
        M1, a0 = C.double() / float(TS[0]), c["alpha0"]
        Y = (a0 + 1) / float(TS[1]) * Z - a0 * torch.outer(M1, M1 @ d["Omega"])
        Q, _ = torch.linalg.qr(Y)
        B = torch.linalg.solve((Q.t() @ d["Omega"]).t(), (Q.t() @ Y).t()).t()
        lam, E = torch.linalg.eigh((B + B.t()) / 2)
        ev = lam.flip(0)[:K]
        W = _signed(Q @ E.flip(1)[:, :K]) / ev.sqrt()
        W0 = d["W"].double()
        Phi = (W.t() @ W0) @ torch.linalg.solve(W0.t() @ W0, d["Phi"].double())
        m1 = W.t() @ M1
        Phi, losses = _pass64(c, d, W, m1, Phi)
        return {"Phi": Phi, "losses": losses, "W": W, "m1": m1, "ev": ev}
    if kind == "sketch":
        return {"Z": _sketch(d["csr"], d["Omega"])[0], "C": None, "TS": None}
    if kind == "topics":
        W, Phi = d["W"].double(), d["Phi"].double()
        n2 = (Phi * Phi).sum(dim=0)
        mu = (W @ torch.linalg.solve(W.t() @ W, Phi) * n2).clamp_(min=0)
        total = mu.sum(dim=0)
        alpha = n2 ** -3
        return {"mu": mu / torch.where(total > 0, total, 1.0), "alpha": alpha / alpha.sum()}
    mu, alpha = d["mu32"].double(), d["alpha"].double()
    theta, gamma = [], []
    for a in range(0, c["docs"], 20000):
        b = min(c["docs"], a + 20000)
        lo, hi = int(d["csr"][0][a]), int(d["csr"][0][b])
        doc, word, f = _rows((d["csr"][0][a:b + 1], d["csr"][1][lo:hi], d["csr"][2][lo:hi]))
        L = torch.zeros(b - a, dtype=torch.float64, device=GPU).index_add_(0, doc, f)
        gm, rows = alpha + L[:, None] / K, mu[word]
        for _ in range(c["iters"]):
            e = torch.digamma(gm)
            p = rows * torch.exp(e - e.max(dim=1, keepdim=True).values)[doc]
            total = p.sum(dim=1, keepdim=True)
            gm = alpha + torch.zeros_like(gm).index_add_(0, doc, f[:, None] * p / torch.where(total > 0, total, 1.0))
        gamma.append(gm)
        theta.append(gm / gm.sum(dim=1, keepdim=True))
    return {"theta": torch.cat(theta), "gamma": torch.cat(gamma)}
