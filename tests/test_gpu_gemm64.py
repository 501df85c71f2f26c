"""C = A B in exact slices where a column of A is all zero (a word without pairs):
the other columns keep their rows' scales."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SRC = r"""
#include "gemm64.cuh"
extern "C" int run(const double *A, const double *B, double *C, int M, int N, int K, int *e) {
  int *ck = e, *ea = e + K, *eb = ea + M;
  cudaMemset(e, 0x80, sizeof(int) * (K + M + N));
  k_col_exp<true><<<dim3((K + 31) / 32, 1), 256>>>(A, K, M, K, M, (const int *)nullptr, ck);
  k_row_exp<<<(M + 7) / 8, 256>>>(A, K, M, K, ck, ea);
  k_col_exp<false><<<dim3((N + 31) / 32, 1), 256>>>(B, N, K, N, K, ck, eb);
  g64_launch<false, false, false>(A, K, B, N, C, N, M, N, K, 1, ea, eb, ck, (cudaStream_t)0);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def product(tmp_path_factory):
    from paper_2511_07809_gb300 import _build

    d = tmp_path_factory.mktemp("gemm64")
    (d / "run.cu").write_text(SRC)
    subprocess.run([_build.NVCC, "-shared", str(d / "run.cu"), "-o", str(d / "run.so")] + _build._flags(), check=True,
                   capture_output=True)
    f = ctypes.CDLL(str(d / "run.so")).run
    f.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int] * 3 + [ctypes.c_void_p]

    def run(A, B):
        (M, K), N = A.shape, B.shape[1]
        a, b = torch.tensor(A, device="cuda"), torch.tensor(B, device="cuda")
        c = torch.full((M, N), 7.0, dtype=torch.float64, device="cuda")
        e = torch.zeros(K + M + N, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert f(a.data_ptr(), b.data_ptr(), c.data_ptr(), M, N, K, e.data_ptr()) == 0
        return c.cpu().numpy()

    return run


@pytest.mark.parametrize("zero", [0, 1, 5])
@pytest.mark.parametrize("M,K,N", [(64, 64, 64), (100, 130, 33), (7, 40, 66)])
def test_rows_keep_their_scale(product, M, K, N, zero):
    rng = np.random.default_rng(M + zero)
    A = rng.standard_normal((M, K)) * 2.0 ** -rng.integers(0, 40, M)[:, None]
    A[0] = rng.standard_normal(K)
    A[:, rng.choice(K, zero, replace=False)] = 0.0
    B = rng.standard_normal((K, N))
    C = product(A, B)
    ref = (A.astype(np.longdouble) @ B.astype(np.longdouble)).astype(np.float64)
    # each term to 2^-53 of its row's and column's largest magnitudes (the term's column scaled to its own largest
    # first, at most 2^2 above 1 here), dropped digit orders as much again
    cs = np.abs(A).max(axis=0)
    row = np.abs(A / np.where(cs > 0, cs, 1.0)).max(axis=1)[:, None]
    col = np.abs(B * cs[:, None]).max(axis=0)[None, :]
    assert (np.abs(C - ref) <= 2.0 ** -53 * 8 * K * row * col).all()
