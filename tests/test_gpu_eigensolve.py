"""The grid-wide eigensolve behind the online whitening: planted problems whose
answer is known to FP64 rounding, alone and beside other work on the GPU."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

V, D, A0 = 600, 20, 1.0


def _planted(r):
    """Statistics of an M2 with r known eigenpairs, and an Omega that sees each of them alike: Omega = U O with O
    orthogonal, so that U^T Omega has condition 1 and Y = M2 Omega that of the spectrum, 1e3."""
    rng = np.random.default_rng(r)
    U = np.linalg.qr(rng.standard_normal((V, r)))[0]
    Om = U @ np.linalg.qr(rng.standard_normal((r, r)))[0]
    lam = np.geomspace(1.0, 1e-3, r) * np.where(np.arange(r) % 3 == 2, -1.0, 1.0)
    C = rng.integers(1, 100, V)
    M1 = C / C.sum()
    Z = ((U * lam) @ (U.T @ Om) + A0 * np.outer(M1, M1 @ Om)) * 1000 / (A0 + 1.0)
    return U, Om, lam, C, M1, Z


def _check(t, U, lam, M1, r):
    W, m1, ev = t.get_whitening()
    W = W.cpu().numpy().astype(np.float64)
    top = np.sort(lam)[::-1][:D]
    # FP64 rounding of sums over r terms times the condition of Y
    bound = 2.0 ** -52 * 64 * r * 1e3
    assert np.abs(ev - top).max() <= bound, (np.abs(ev - top).max(), bound)
    # W^T M2 W = I: besides that the columns of W rounded to FP32, each way
    G = W.T @ ((U * lam) @ (U.T @ W))
    assert np.abs(G - np.eye(D)).max() <= 2.0 ** -24 * 4 * np.sqrt(top[0] / top[-1]) + bound / top[-1]
    assert np.abs(m1.cpu().numpy() - W.T @ M1).max() <= 2.0 ** -22 * np.abs(W).max()


@pytest.mark.parametrize("r", [32, 34, 64, 66, 130, 216, 258, 512])
def test_eigensolve(lib, r):
    U, Om, lam, C, M1, Z = _planted(r)
    t = lib.TLDA(V, D, alpha0=A0, max_batch=64)
    t.online_begin(torch.tensor(Om))
    t.online_set_sketch(torch.tensor(Z), torch.tensor(C), torch.tensor([int(C.sum()), 1000, 0]))
    t.online_whiten()
    _check(t, U, lam, M1, r)
    t.close()


@pytest.mark.parametrize("r", [66, 216])
def test_eigensolve_beside_other_work(lib, r):
    """Blocks of a round held up by another stream's kernels on their SMs: every tile still rotates by the same
    angles."""
    U, Om, lam, C, M1, Z = _planted(r)
    t = lib.TLDA(V, D, alpha0=A0, max_batch=64)
    t.online_begin(torch.tensor(Om))
    t.online_set_sketch(torch.tensor(Z), torch.tensor(C), torch.tensor([int(C.sum()), 1000, 0]))
    side = torch.cuda.Stream()
    x = torch.rand(1 << 16, device="cuda")
    side.wait_stream(torch.cuda.current_stream())
    for _ in range(10):
        with torch.cuda.stream(side):
            for _ in range(200):
                x = torch.sin(x)
        t.online_whiten()
        _check(t, U, lam, M1, r)
    torch.cuda.synchronize()
    t.close()
