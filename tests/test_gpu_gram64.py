"""Gram matrices in exact slices where a column's few large entries carry it (the whitening
of a Zipf vocabulary): as near to 64 bits as a few roundings of the result."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SRC = r"""
#include "gemm64.cuh"
extern "C" int gram(const double *A, double *C, int K, int N, int splits, int *e) {
  cudaMemset(e, 0x80, sizeof(int) * N);
  cudaMemset(C, 0, sizeof(double) * N * N);
  k_col_exp<false><<<dim3((N + 31) / 32, 1), 256>>>(A, N, K, N, K, (const int *)nullptr, e);
  g64_launch<true, true, true>(A, N, A, N, C, N, N, N, K, splits, e, e, (const int *)nullptr, (cudaStream_t)0);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("V,K,splits", [(5285, 19, 1), (5285, 19, 8), (12865, 70, 4), (100, 64, 1)])
def test_gram_of_peaked_columns(tmp_path, V, K, splits):
    from paper_2511_07809_gb300 import _build

    (tmp_path / "run.cu").write_text(SRC)
    subprocess.run([_build.NVCC, "-shared", str(tmp_path / "run.cu"), "-o", str(tmp_path / "run.so")] + _build._flags(),
                   check=True, capture_output=True)
    f = ctypes.CDLL(str(tmp_path / "run.so")).gram
    f.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int] * 3 + [ctypes.c_void_p]
    rng = np.random.default_rng(V + K)
    p = np.arange(1, V + 1) ** -1.1
    w = rng.standard_gamma(np.array([rng.permutation(0.05 * V * p / p.sum()) for _ in range(K)]))
    mu = (w / w.sum(axis=1, keepdims=True)).T
    lam, E = np.linalg.eigh(mu.T @ mu / K)
    A = (mu @ E / (lam * np.sqrt(K))).astype(np.float32).astype(np.float64)
    a = torch.tensor(A, device="cuda")
    c = torch.zeros((K, K), dtype=torch.float64, device="cuda")
    e = torch.zeros(K, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert f(a.data_ptr(), c.data_ptr(), V, K, splits, e.data_ptr()) == 0
    ref = A.T.astype(np.longdouble) @ A.astype(np.longdouble)
    err = np.linalg.norm((c.cpu().numpy() - ref).astype(np.float64)) / np.linalg.norm(ref.astype(np.float64))
    assert err <= 2.0 ** -51, err  # 28 digit products a term give 5e-15 here, plain FP64 sums some 4e-16
