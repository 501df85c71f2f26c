// Moments and whitening (section "Computing the Centered Cumulants", appendix
// "Uncentered cumulants", section "Online Decomposition of the Second
// Moment") and topic recovery (section "Recovering the Topic Model
// Parameters"), on the device.
//
//  ACCUMULATE  exact integer statistics of each chunk: C_m, T, S2, S3 (int64)
//              and the pair counts P = sum_d (f_d f_d^T - diag f_d), held as a
//              dense V x V FP64 matrix of exact integers (atomic adds of
//              integers below 2^53 are order independent).
//  FINALIZE    M1 = C/T, M2 = (alpha0+1) P/S2 - alpha0 M1 M1^T; top-D
//              eigenpairs by randomised subspace iteration (FP32 products,
//              FP64 CholeskyQR), FP64 Rayleigh-Ritz with a cyclic Jacobi
//              eigensolver over the grid, W = U Lambda^-1/2, m1 = W^T M1.
//              FP64 products run on the tensor cores in exact slices (gemm64.cuh).
//  unwhiten    mu_i = ||phi_i||^2 W (W^T W)^-1 phi_i, alpha_i ~ ||phi_i||^-6,
//              clip at 0, normalise (FP64).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <functional>
#include <type_traits>
#include <vector>

#include "gemm64.cuh"
#include "scan.cuh"
#include "tlda_internal.h"

using namespace tlda;

namespace {

constexpr int kMaxFitV = 65536;
constexpr size_t kKeepTopics = size_t(32) << 20;   // bytes of topics that a context keeps room for
constexpr int kOversample = 16;                    // columns of the fit's subspace beyond D
constexpr int kMaxRitz = kMaxDim + kOversample;    // largest order of the dense FP64 kernels

// ------------------------------------------------------------------ scan + pairs
// One warp per document.  Only the pairs on or below the diagonal of P are
// added (the words ascend within a document); k_m2_mirror fills in the rest.
__global__ void k_fit_accumulate(tlda_csr b, int V, double *P, unsigned long long *C,
                                 unsigned long long *TS, int *err) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= b.n_docs) return;
  const int lo = b.indptr[warp], hi = b.indptr[warp + 1];
  if (lo < 0 || hi < lo) {
    if (lane == 0) atomicOr(err, 1);
    return;
  }
  const int u = hi - lo;
  bool bad = false;
  long long L = 0;
  for (int j = lo + lane; j < hi; j += 32) {
    const int m = b.indices[j], f = b.counts[j];
    if (m < 0 || m >= V || f <= 0 || (j > lo && m <= b.indices[j - 1])) bad = true;
    else L += f;
  }
  if (__any_sync(0xffffffffu, bad)) {
    if (lane == 0) atomicOr(err, 1);
    return;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  if (lane == 0) {
    atomicAdd(TS + 0, (unsigned long long)L);
    atomicAdd(TS + 1, (unsigned long long)(L * (L - 1)));
    atomicAdd(TS + 2, (unsigned long long)(L * (L - 1) * (L - 2)));
  }
  for (int j = lo + lane; j < hi; j += 32) atomicAdd(C + b.indices[j], (unsigned long long)b.counts[j]);
  // pair t of the lower triangle by rows: row x holds t = x(x+1)/2 .. x(x+1)/2 + x
  const long long np = (long long)u * (u + 1) / 2;
  int x = 0;
  long long row = 0;  // first pair of row x
  for (long long t = lane; t < np; t += 32) {
    while (t > row + x) {
      row += x + 1;
      ++x;
    }
    const int y = (int)(t - row);
    const int ma = b.indices[lo + x], mb = b.indices[lo + y];
    const long long fa = b.counts[lo + x], fb = b.counts[lo + y];
    const long long v = fa * fb - (x == y ? fa : 0);
    if (v) atomicAdd(P + (long long)ma * V + mb, (double)v);
  }
}

// ------------------------------------------------------------------ products
// FP32: C[M x N] = A[M x Kd] B[Kd x N] (row-major, any pitch), FFMA.  Tiles of
// 16 TM rows x 16 TN columns, TM x TN outputs a thread, so that N = 66 or 116
// columns (D + 16) waste at most 15 of a tile; slabs of 32 terms pass through
// three stages of shared memory by cp.async (16 bytes a piece where A's rows
// allow it).  Few row tiles leave SMs idle, so the terms are split over
// blockIdx.z into partial products (sgemm_splits), summed in order by
// k_sgemm_sum.  M2 Q at V = 5000, N = 66: 122 us (286 with 64 x 64 tiles and no
// split; the FFMA rate alone would allow 52 with the tile's padding); Q L^-T, 66
// terms in 32-row tiles: 9 us (28 in 128-row tiles, 40 blocks).
constexpr int kSgBk = 32, kSgStages = 3;
template <int TM, int TN>
constexpr int sgemm_smem() { return kSgStages * (16 * TM * (kSgBk + 4) + kSgBk * 16 * TN) * 4; }

template <int TM, int TN, bool WIDE>
__global__ void __launch_bounds__(256) k_sgemm(const float *__restrict__ A, int lda, const float *__restrict__ B, int ldb,
                                               float *__restrict__ C, int ldc, int M, int N, int Kd, int chunk,
                                               long long cstride) {
  constexpr int BM = 16 * TM, BN = 16 * TN, BK = kSgBk, LDA = BK + 4, STAGE = BM * LDA + BK * BN;
  extern __shared__ __align__(16) float sg_sm[];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int kb = blockIdx.z * chunk, ke = min(Kd, kb + chunk), slabs = (ke - kb + BK - 1) / BK;
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  auto request = [&](int q) {
    if (q < slabs) {
      float *As = sg_sm + (q % kSgStages) * STAGE, *Bs = As + BM * LDA;
      const int k0 = kb + q * BK;
      if (WIDE) {  // kb, ke, lda multiples of 4 and A on 16 bytes
#pragma unroll
        for (int i = 0; i < BM * BK / 1024; ++i) {
          const int e = tid + i * 256, r = e >> 3, k = (e & 7) * 4;
          const bool in = k0 + k < ke && m0 + r < M;
          const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(As + r * LDA + k));
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(in ? A + (long long)(m0 + r) * lda + k0 + k : A),
                       "r"(in ? 16 : 0)
                       : "memory");
        }
      } else {
#pragma unroll
        for (int i = 0; i < BM * BK / 256; ++i) {
          const int e = tid + i * 256, r = e >> 5, k = e & 31;
          const bool in = k0 + k < ke && m0 + r < M;
          g64_cp(As + r * LDA + k, in ? A + (long long)(m0 + r) * lda + k0 + k : A, in);
        }
      }
#pragma unroll
      for (int i = 0; i < BK * BN / 256; ++i) {
        const int e = tid + i * 256, k = e / BN, c = e % BN;
        const bool in = k0 + k < ke && n0 + c < N;
        g64_cp(Bs + k * BN + c, in ? B + (long long)(k0 + k) * ldb + n0 + c : B, in);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  request(0);
  request(1);
  for (int q = 0; q < slabs; ++q) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    request(q + 2);  // into the stage of slab q - 1, which has been read
    const float *As = sg_sm + (q % kSgStages) * STAGE + ty * LDA, *Bs = sg_sm + (q % kSgStages) * STAGE + BM * LDA;
#pragma unroll 2
    for (int k = 0; k < BK; k += 4) {
      float4 x[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) x[i] = *reinterpret_cast<const float4 *>(As + 16 * i * LDA + k);  // a warp's two rows: other banks
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float br[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) br[j] = Bs[(k + u) * BN + tx + 16 * j];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const float xi = u == 0 ? x[i].x : u == 1 ? x[i].y : u == 2 ? x[i].z : x[i].w;
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(xi, br[j], acc[i][j]);
        }
      }
    }
  }
  float *c = C + blockIdx.z * cstride;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int r = m0 + ty + 16 * i;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int n = n0 + tx + 16 * j;
      if (r < M && n < N) c[(long long)r * ldc + n] = acc[i][j];
    }
  }
}

__global__ void k_sgemm_sum(const float *part, int splits, long long n, float *C) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  float v = part[e];
  for (int s = 1; s < splits; ++s) v += part[s * n + e];
  C[e] = v;
}

// Splits of the terms: about two tiles per SM, at least 256 terms each.
int sgemm_splits(int M, int N, int Kd, int sms) {
  const int tiles = ((M + 127) / 128) * ((N + 127) / 128);
  return std::max(1, std::min(2 * sms / tiles, Kd / 256));
}

template <int TM, int TN>
void sgemm_launch(const float *A, int lda, const float *B, int ldb, float *out, int M, int N, int Kd, int chunk, int splits,
                  cudaStream_t s) {
  static SmemLimit lim[2];
  lim[0].raise((const void *)k_sgemm<TM, TN, true>, sgemm_smem<TM, TN>());
  lim[1].raise((const void *)k_sgemm<TM, TN, false>, sgemm_smem<TM, TN>());
  const dim3 g((N + 16 * TN - 1) / (16 * TN), (M + 16 * TM - 1) / (16 * TM), splits);
  const bool wide = lda % 4 == 0 && Kd % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;  // chunk is a multiple of 32
  if (wide) k_sgemm<TM, TN, true><<<g, 256, sgemm_smem<TM, TN>(), s>>>(A, lda, B, ldb, out, N, M, N, Kd, chunk, (long long)M * N);
  else k_sgemm<TM, TN, false><<<g, 256, sgemm_smem<TM, TN>(), s>>>(A, lda, B, ldb, out, N, M, N, Kd, chunk, (long long)M * N);
}

// part: splits x M x N floats when there is more than one split (C then is M x N).
// Products of few terms (Q L^-T, at most kMaxRitz) take tiles of 32 rows, for more
// blocks; with many terms 128 rows are ahead also where they are not split (the
// fit's milliseconds in 32-row tiles and these: V = 30,000 and D = 100 310 -> 241,
// V = 20,000 and D = 40 89.2 -> 85.8, V = 12,000 and D = 150 86.0 -> 84.8; V =
// 20,000 and D = 100, five tiles more than SMs, 155.0 -> 155.5).
void sgemm(const float *A, int lda, const float *B, int ldb, float *C, int M, int N, int Kd, float *part, int splits,
           cudaStream_t s) {
  const int nt = (N + 127) / 128, tn = (N + 16 * nt - 1) / (16 * nt);
  const int chunk = ((Kd + splits - 1) / splits + kSgBk - 1) / kSgBk * kSgBk;
  splits = (Kd + chunk - 1) / chunk;
  float *out = splits > 1 ? part : C;
  const bool tall = Kd >= 2 * kMaxDim || splits > 1;
#define TLDA_SGEMM(TNv)                                                                         \
  case TNv:                                                                                     \
    if (tall) sgemm_launch<8, TNv>(A, lda, B, ldb, out, M, N, Kd, chunk, splits, s);            \
    else sgemm_launch<2, TNv>(A, lda, B, ldb, out, M, N, Kd, chunk, splits, s);                 \
    break;
  switch (tn) {
    TLDA_SGEMM(1) TLDA_SGEMM(2) TLDA_SGEMM(3) TLDA_SGEMM(4) TLDA_SGEMM(5) TLDA_SGEMM(6) TLDA_SGEMM(7) TLDA_SGEMM(8)
  }
#undef TLDA_SGEMM
  if (splits > 1) {
    const long long n = (long long)M * N;
    k_sgemm_sum<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(part, splits, n, C);
  }
}

// Exponents of the operands of the FP64 products (gemm64.cuh): V rows, V terms,
// then two sets of up to 2 kMaxDim columns.
constexpr int kExpCols = 2 * kMaxDim;

template <bool FIN, class T>
void col_exp(const T *x, int ld, int rows, int cols, const int *add, int *e, cudaStream_t s) {
  const int slab = std::max(64, (rows + 63) / 64);
  cudaMemsetAsync(e, 0x80, sizeof(int) * cols, s);
  k_col_exp<FIN, T><<<dim3((cols + 31) / 32, (rows + slab - 1) / slab), 256, 0, s>>>(x, ld, rows, cols, slab, add, e);
}

// Splits of the terms of an FP64 product: one block per SM runs, so the time
// goes with the waves of blocks over the splits.
int gemm64_splits(int tiles, int Kd, int sms) {
  const int folds = (Kd + kG64Fold - 1) / kG64Fold;
  int best = 1;
  double cost = 1e30;
  for (int S = 1; S <= folds && S <= 64; ++S) {
    const int waves = (tiles * S + sms - 1) / sms, per = (folds + S - 1) / S;
    const double c = (double)waves * (per + 0.5);  // a block's start and its sums into C: about half a fold's time
    if (c < cost) {
      cost = c;
      best = S;
    }
  }
  return best;
}

// C[M x N] = A^T B (FP64), A: Kd x M, B: Kd x N.  exps: ctx->g64_exp.
template <class TA, class TB>
void gemm_tn64(const TA *A, int lda, const TB *B, int ldb, double *C, int ldc, int M, int N, int Kd, int *exps, int V,
               int sms, cudaStream_t s) {
  cudaMemsetAsync(C, 0, sizeof(double) * (size_t)M * ldc, s);
  int *eA = exps + 2 * (size_t)V, *eB = eA + kExpCols;
  const int tm = (M + kG64Tile - 1) / kG64Tile, tn = (N + kG64Tile - 1) / kG64Tile;
  col_exp<false>(A, lda, Kd, M, nullptr, eA, s);
  if (static_cast<const void *>(A) == static_cast<const void *>(B) && lda == ldb && M == N && sizeof(TA) == sizeof(TB)) {
    g64_launch<true, true, true>(A, lda, B, ldb, C, ldc, M, N, Kd, gemm64_splits(tm * (tm + 1) / 2, Kd, sms), eA, eA,
                                 nullptr, s);
  } else {
    col_exp<false>(B, ldb, Kd, N, nullptr, eB, s);
    g64_launch<true, true, false>(A, lda, B, ldb, C, ldc, M, N, Kd, gemm64_splits(tm * tn, Kd, sms), eA, eB, nullptr, s);
  }
}

// C[M x N] = A B (FP64), A: M x Kd (M, Kd <= V), B: Kd x N.
template <class TA>
void gemm_nn64(const TA *A, int lda, const double *B, int ldb, double *C, int ldc, int M, int N, int Kd, int *exps, int V,
               int sms, cudaStream_t s) {
  int *eA = exps, *ck = exps + V, *eB = exps + 2 * (size_t)V;
  col_exp<true>(A, lda, M, Kd, nullptr, ck, s);
  k_row_exp<TA><<<(M + 7) / 8, 256, 0, s>>>(A, lda, M, Kd, ck, eA);
  col_exp<false>(B, ldb, Kd, N, ck, eB, s);
  const int tiles = ((M + kG64Tile - 1) / kG64Tile) * ((N + kG64Tile - 1) / kG64Tile);
  const int splits = gemm64_splits(tiles, Kd, sms);
  if (splits > 1) {
    cudaMemsetAsync(C, 0, sizeof(double) * (size_t)M * ldc, s);
    g64_launch<false, true, false>(A, lda, B, ldb, C, ldc, M, N, Kd, splits, eA, eB, ck, s);
  } else {
    g64_launch<false, false, false>(A, lda, B, ldb, C, ldc, M, N, Kd, 1, eA, eB, ck, s);
  }
}

// y[j] += sum over a slab of rows of x[m] Q[m][j] (FP64; y zeroed before): one
// block per 32 columns and slab.
__global__ void __launch_bounds__(256) k_vec_tn64(const double *x, const double *Q, int rows, int cols, int slab, double *y) {
  __shared__ double red[8][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  const int r0 = blockIdx.y * slab, r1 = min(rows, r0 + slab);
  double v = 0.0;
  if (c < cols)
    for (int r = r0 + w; r < r1; r += 8) v = fma(x[r], Q[(long long)r * cols + c], v);
  red[w][lane] = v;
  __syncthreads();
  if (w == 0 && c < cols) {
#pragma unroll
    for (int q = 1; q < 8; ++q) v += red[q][lane];
    atomicAdd(y + c, v);
  }
}

void vec_tn64(const double *x, const double *Q, int rows, int cols, double *y, cudaStream_t s) {
  const int slab = std::max(32, (rows + 63) / 64);
  cudaMemsetAsync(y, 0, sizeof(double) * cols, s);
  k_vec_tn64<<<dim3((cols + 31) / 32, (rows + slab - 1) / slab), 256, 0, s>>>(x, Q, rows, cols, slab, y);
}

// out (D x K) = R X with R FP64 (D x D), plain FP64 sums, one block per row: the
// products of small triangular factors, whose entries may differ in scale by
// more than exact slices hold.  scale (K) multiplies the columns when given.
template <class TX, class TO>
__global__ void __launch_bounds__(256) k_small_nn(const double *R, const TX *X, int D, int K, const double *scale, TO *out) {
  __shared__ double g[kMaxDim];
  const int r = blockIdx.x;
  for (int j = threadIdx.x; j < D; j += 256) g[j] = R[r * D + j];
  __syncthreads();
  for (int i = threadIdx.x; i < K; i += 256) {
    double v = 0.0;
#pragma unroll 8
    for (int j = 0; j < D; ++j) v = fma(g[j], (double)X[j * K + i], v);
    out[r * K + i] = (TO)(scale ? v * scale[i] : v);
  }
}

// ------------------------------------------------------------------ elementwise helpers
// The upper half of P (32 x 32 tiles, read below the diagonal) and the FP32
// M2 = sP P - a0 M1 M1^T in both halves.
__global__ void __launch_bounds__(256) k_m2_mirror(double *P, const double *M1, int V, double sP, double a0, float *M2) {
  const int by = blockIdx.y, bx = blockIdx.x;
  if (bx > by) return;
  __shared__ double t[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = by * 32 + ty + 8 * q, j = bx * 32 + tx;
    t[ty + 8 * q][tx] = (i < V && j < V) ? P[(long long)i * V + j] : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = ty + 8 * q;
    int i = by * 32 + r, j = bx * 32 + tx;
    const bool low = bx < by || tx <= r;  // the entry below the diagonal that this one equals
    if (i < V && j < V) {
      const double v = low ? t[r][tx] : t[tx][r];
      M2[(long long)i * V + j] = (float)(sP * v - a0 * M1[i] * M1[j]);
      if (!low) P[(long long)i * V + j] = v;
    }
    if (bx < by) {
      i = bx * 32 + r, j = by * 32 + tx;
      if (i < V && j < V) {
        const double v = t[tx][r];
        P[(long long)i * V + j] = v;
        M2[(long long)i * V + j] = (float)(sP * v - a0 * M1[i] * M1[j]);
      }
    }
  }
}

__global__ void k_m1(const unsigned long long *C, const unsigned long long *TS, int V, double *M1) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < V) M1[m] = (double)C[m] / (double)TS[0];
}

__device__ inline unsigned long long splitmix64(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

// Gaussian start block Omega (V x r), Box-Muller on a counter hash.
__global__ void k_gauss(float *O, long long n, unsigned long long seed) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const unsigned long long h1 = splitmix64(seed ^ (2 * e)), h2 = splitmix64(seed ^ (2 * e + 1) ^ 0x5851F42D4C957F2Dull);
  const double u1 = ((h1 >> 11) + 0.5) * (1.0 / 9007199254740992.0);
  const double u2 = (h2 >> 11) * (1.0 / 9007199254740992.0);
  O[e] = (float)(sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2));
}

__global__ void k_d2f(const double *x, float *y, long long n) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) y[e] = (float)x[e];
}

// ------------------------------------------------------------------ small dense FP64
__global__ void k_transpose_rr(const double *A, int r, double *AT) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= r * r) return;
  const int i = e / r, j = e % r;
  AT[j * r + i] = A[e];
}

// Control block of the grid-wide Jacobi: the grid barrier's arrival counter,
// an abort flag, the sweep count, and each block's partial sums of the squared
// off-diagonal and total entries (two slots, by sweep parity).
constexpr int kJacThreads = 256, kJacMaxGrid = 256;
struct JacCtl {
  unsigned bar;
  int abort;
  int sweeps;
  int pad;
  double part[2][2][kJacMaxGrid];
};

__device__ __forceinline__ unsigned jac_ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier of a cooperative launch (every block resident): a release
// increment of the arrival counter, then acquire loads until it reaches
// `target`; bounded to about a second; false if it expired here or any block
// flagged an abort.
__device__ bool jac_sync(JacCtl *ctl, unsigned target, int *s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->bar) : "memory");
    const long long t0 = clock64();
    // the abort flag and the bound are looked at every 16th poll: each look is
    // a round trip to L2 of its own
    for (int poll = 1; jac_ld_acquire(&ctl->bar) < target; ++poll) {
      if (poll & 15) continue;
      if (*reinterpret_cast<volatile int *>(&ctl->abort)) {
        ok = 0;
        break;
      }
      if (clock64() - t0 > 2000000000ll) {
        atomicExch(&ctl->abort, 1);
        ok = 0;
        break;
      }
    }
    *reinterpret_cast<volatile int *>(s_ok) = ok;
  }
  __syncthreads();
  return *reinterpret_cast<volatile int *>(s_ok) != 0;
}

// FP64 to FP32 and back on the integer units, toward zero: a conversion takes
// the FP64 pipe 65 cycles.  Outside FP32's normal range: 0 below, infinity above.
// off: 896 plus the exponent of a power of two that x is divided by (positive).
__device__ __forceinline__ float seed_f32(double x, int off = 896) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff) - off;  // FP32 exponent field
  const uint32_t m = (uint32_t)(b >> 29) & 0x7fffffu, s = (uint32_t)(b >> 32) & 0x80000000u;
  return __uint_as_float(s | (e <= 0 ? 0u : e >= 255 ? 0x7f800000u : ((uint32_t)e << 23) | m));
}
__device__ __forceinline__ double widen_f32(float x) {  // finite; below FP32's normal range: 0
  const uint32_t b = __float_as_uint(x), e = (b >> 23) & 0xffu;
  const long long s = (long long)(b & 0x80000000u) << 32;
  return __longlong_as_double(e == 0 ? s : s | ((long long)(e + 896) << 52) | ((long long)(b & 0x7fffffu) << 29));
}

// 1/d: FP32, then one third-order step (d in FP32's normal range, else divided).
__device__ __forceinline__ double recip64(double d) {
  const float f = __frcp_rn(seed_f32(d)), a = fabsf(f);
  if (!(a > 1e-37f && a < 1e37f)) return 1.0 / d;
  const double q = widen_f32(f), e = fma(-d, q, 1.0);
  return fma(q, fma(e, e, e), q);
}

// Slot of the round-robin ordering: slot 0 holds index 0, the others rotate.
__device__ __forceinline__ int jac_slot(int slot, int round, int r) {
  const int x = slot - 1 + round;  // below 2 (r - 1)
  return slot == 0 ? 0 : 1 + (x >= r - 1 ? x - (r - 1) : x);
}

// Indices p < q of pair k in a round.
__device__ __forceinline__ void jac_pair(int k, int round, int r, int &p, int &q) {
  const int a = jac_slot(k, round, r), b = jac_slot(r - 1 - k, round, r);
  p = min(a, b);
  q = max(a, b);
}

// Cyclic Jacobi for a symmetric r x r FP64 matrix A0 (r even, global memory,
// overwritten; A1: as much scratch), round-robin ordering so each round applies r/2 disjoint
// rotations in parallel (Golub & Van Loan, "Matrix Computations", sec. 8.5,
// parallel ordering).  Rotation of pair (p, q): tau = (a_qq - a_pp)/(2 a_pq),
// t = sign(tau)/(|tau| + sqrt(1 + tau^2)), c = 1/sqrt(1 + t^2), s = t c.
// Because the rotations of one round are disjoint, A <- J^T A J is applied in
// one pass over the 2 x 2 blocks (pair k rows, pair l columns), each block
// rotated on the left by pair k and on the right by pair l; the eigenvectors
// are kept as rows, Et <- J^T Et.  The rotations' entries are read by every tile
// that holds one of the pairs while the diagonal tiles rotate them, so a round
// reads A from one copy and writes it, whole, to the other; an entry of Et has one
// reader and writer a round.  Et starts as I; on return eval[i] = A_ii and
// row i of Et is its eigenvector.  Sweeps stop when the off-diagonal mass is
// below 1e-26 r^2 of the total, i.e. entries near 1e-13 of the scale (or after
// max_sweeps).
// A round is bound by its latency: one grid barrier, one L2 round trip, and the
// FP64 pipe, which takes 2 operations a clock per SM.  So the 2 x 2 blocks are
// dealt as tiles of bt x bt pairs over T x T thread blocks: a block needs the
// rotations of its 2 bt pairs only, not of all r/2; its entries are requested
// before the rotations are computed; and the angle is found in FP32 and made good
// to 1e-14 by one Newton step whose rest is FP64, with c = (1 - h^2)/(1 + h^2) and
// s = 2 h/(1 + h^2) for the tangent h of its half (an FP64 division or square root
// takes 430 to 680 cycles here): the rotation is orthogonal to FP64 rounding.
// FP32 takes the entries relative to the norm of A, so that any scale will do: an
// entry 2^-126 below the norm is left as it is, far under the stopping rule.
// Without the step an r = 216 solve takes 0.45 ms less of 6.9, but then the entries
// that the last sweep leaves under the stopping rule, and with them the
// eigenvectors at 1e-8, are others than with exact angles.
__global__ void __launch_bounds__(kJacThreads) k_jacobi(double *A0, double *A1, int r, double *__restrict__ Et,
                                                       double *__restrict__ eval, int max_sweeps,
                                                       JacCtl *ctl) {
  __shared__ double cs[2][kMaxRitz / 2], sn[2][kMaxRitz / 2];  // rows' pairs, columns' pairs of this block
  __shared__ double red_o[kJacThreads / 32], red_t[kJacThreads / 32];
  __shared__ int s_ok, s_done, s_off;
  const int G = gridDim.x, tid = threadIdx.x, nt = blockDim.x;
  const int gt = blockIdx.x * nt + tid, gn = G * nt;
  const int h = r / 2, rr = r * r;
  int T = 1;
  while ((T + 1) * (T + 1) <= G) ++T;
  const int bt = (h + T - 1) / T, ti = blockIdx.x / T, tj = blockIdx.x % T;
  const int ka = min(h, ti * bt), kn = blockIdx.x < T * T ? min(h, ka + bt) - ka : 0;
  const int la = min(h, tj * bt), ln = min(h, la + bt) - la;
  const int ja = (int)((long long)r * tj / T), jn = (int)((long long)r * (tj + 1) / T) - ja;  // columns of Et
  const int nb = kn * ln, ne = kn * jn;
  // this thread's first two 2 x 2 blocks and four eigenvector pairs, in every round
  int bk[2] = {}, bl[2] = {}, ek[4] = {}, ej[4] = {};
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (tid + u * nt < nb) bk[u] = (tid + u * nt) / ln, bl[u] = (tid + u * nt) % ln;
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (tid + u * nt < ne) ek[u] = (tid + u * nt) / jn, ej[u] = (tid + u * nt) % jn;
  unsigned nbar = 0;
  double *A = A0, *An = A1;  // this round's copy, the next one's
  for (int e = gt; e < rr; e += gn) {
    const int i = e / r, j = e % r;
    if (i < j) {
      const double v = 0.5 * (A[i * r + j] + A[j * r + i]);
      A[i * r + j] = v;
      A[j * r + i] = v;
    }
    Et[e] = (i == j) ? 1.0 : 0.0;
  }
  if (!jac_sync(ctl, ++nbar * G, &s_ok)) return;
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    double o = 0.0, t = 0.0;
    for (int e = gt; e < rr; e += gn) {
      const double v = __ldcg(A + e);
      t += v * v;
      if (e / r != e % r) o += v * v;
    }
    for (int m = 16; m > 0; m >>= 1) {
      o += __shfl_xor_sync(0xffffffffu, o, m);
      t += __shfl_xor_sync(0xffffffffu, t, m);
    }
    if ((tid & 31) == 0) {
      red_o[tid >> 5] = o;
      red_t[tid >> 5] = t;
    }
    __syncthreads();
    if (tid == 0) {
      double so = 0.0, st = 0.0;
      for (int w = 0; w < nt / 32; ++w) {
        so += red_o[w];
        st += red_t[w];
      }
      ctl->part[sweep & 1][0][blockIdx.x] = so;
      ctl->part[sweep & 1][1][blockIdx.x] = st;
    }
    if (!jac_sync(ctl, ++nbar * G, &s_ok)) return;
    if (tid < 32) {  // every block sums the partials in the same order
      double so = 0.0, st = 0.0;
      for (int g = tid; g < G; g += 32) {
        so += __ldcg(&ctl->part[sweep & 1][0][g]);
        st += __ldcg(&ctl->part[sweep & 1][1][g]);
      }
      for (int m = 16; m > 0; m >>= 1) {
        so += __shfl_xor_sync(0xffffffffu, so, m);
        st += __shfl_xor_sync(0xffffffffu, st, m);
      }
      if (tid == 0) {
        s_done = so <= 1e-26 * (double)r * r * st;
        s_off = 896 + (((__double2hiint(st) >> 20) & 0x7ff) - 1023) / 2;  // half the exponent of the squared norm
      }
    }
    __syncthreads();
    if (s_done) break;
    const int off = s_off;
    for (int round = 0; round < r - 1; ++round) {
      double x[2][4], ev[4][2];
      int bx[2][4], ei[4][2];
      auto block_at = [&](int k, int l, int (&base)[4]) {
        int pk, qk, pl, ql;
        jac_pair(ka + k, round, r, pk, qk);
        jac_pair(la + l, round, r, pl, ql);
        base[0] = pk * r + pl;
        base[1] = pk * r + ql;
        base[2] = qk * r + pl;
        base[3] = qk * r + ql;
      };
      auto pair_at = [&](int k, int j, int (&base)[2]) {
        int p, q;
        jac_pair(ka + k, round, r, p, q);
        base[0] = p * r + ja + j;
        base[1] = q * r + ja + j;
      };
      // the rotations' entries first: they are waited for first
      const bool mine = tid < kn + ln;
      int p = 0, q = 0;
      if (mine) jac_pair(tid < kn ? ka + tid : la + tid - kn, round, r, p, q);
      double apq = 0.0, app = 0.0, aqq = 0.0;
      if (mine) {
        apq = __ldcg(A + p * r + q);
        app = __ldcg(A + p * r + p);
        aqq = __ldcg(A + q * r + q);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (tid + u * nt < nb) {
          block_at(bk[u], bl[u], bx[u]);
#pragma unroll
          for (int v = 0; v < 4; ++v) x[u][v] = __ldcg(A + bx[u][v]);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (tid + u * nt < ne) {
          pair_at(ek[u], ej[u], ei[u]);
#pragma unroll
          for (int v = 0; v < 2; ++v) ev[u][v] = __ldcg(Et + ei[u][v]);
        }
      auto put_rotation = [&](int at, double apq, double app, double aqq) {
        double c = 1.0, sv = 0.0;
        const float fp = seed_f32(apq, off), fd = seed_f32(aqq - app, off);
        if (fp != 0.f) {
          const float tau = __fdividef(0.5f * fd, fp), f = fabsf(tau);
          const float t = __frcp_rn(f + __fsqrt_rn(fmaf(f, f, 1.f)));
          const float h1 = __fdividef(t, 1.f + __fsqrt_rn(fmaf(t, t, 1.f)));  // tan of half the angle, at most 0.42
          double hh = widen_f32(tau < 0.f ? -h1 : h1);
          // Newton from the rest that this angle would leave (times (1 + h^2)^2)
          const double u = fma(-hh, hh, 1.0), v = 2.0 * hh, uv = u * v, uu = fma(u, u, -v * v);
          const float rest = seed_f32(fma(uu, apq, -uv * (aqq - app)), off);
          const float slope = fmaf(seed_f32(uu), fd, 4.f * seed_f32(uv) * fp);
          hh += widen_f32(__fdividef(0.5f * fmaf(h1, h1, 1.f) * rest, slope));
          const double w = fma(hh, hh, 1.0);
          const double q = recip64(w);
          c = fma(2.0, q, -1.0);
          sv = 2.0 * hh * q;
        }
        const int side = at < kn ? 0 : 1, of = at < kn ? at : at - kn;
        cs[side][of] = c;
        sn[side][of] = sv;
      };
      if (mine) put_rotation(tid, apq, app, aqq);
      for (int w = tid + nt; w < kn + ln; w += nt) {  // a small grid's tiles have more pairs than threads
        jac_pair(w < kn ? ka + w : la + w - kn, round, r, p, q);
        put_rotation(w, __ldcg(A + p * r + q), __ldcg(A + p * r + p), __ldcg(A + q * r + q));
      }
      __syncthreads();
      auto rotate_block = [&](int k, int l, const double (&v)[4], const int (&base)[4]) {
        const double ck = cs[0][k], sk = sn[0][k], cl = cs[1][l], sl = sn[1][l];
        const double a1 = ck * v[0] - sk * v[2], b1 = ck * v[1] - sk * v[3];
        const double c1 = sk * v[0] + ck * v[2], d1 = sk * v[1] + ck * v[3];
        An[base[0]] = cl * a1 - sl * b1;
        An[base[1]] = sl * a1 + cl * b1;
        An[base[2]] = cl * c1 - sl * d1;
        An[base[3]] = sl * c1 + cl * d1;
      };
      auto rotate_pair = [&](int k, const double (&v)[2], const int (&base)[2]) {
        const double c = cs[0][k], sv = sn[0][k];
        Et[base[0]] = c * v[0] - sv * v[1];
        Et[base[1]] = sv * v[0] + c * v[1];
      };
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (tid + u * nt < nb) rotate_block(bk[u], bl[u], x[u], bx[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (tid + u * nt < ne) rotate_pair(ek[u], ev[u], ei[u]);
      // what a small grid leaves over
      for (int w = tid + 2 * nt; w < nb; w += nt) {
        block_at(w / ln, w % ln, bx[0]);
#pragma unroll
        for (int v = 0; v < 4; ++v) x[0][v] = __ldcg(A + bx[0][v]);
        rotate_block(w / ln, w % ln, x[0], bx[0]);
      }
      for (int w = tid + 4 * nt; w < ne; w += nt) {
        pair_at(w / jn, w % jn, ei[0]);
#pragma unroll
        for (int v = 0; v < 2; ++v) ev[0][v] = __ldcg(Et + ei[0][v]);
        rotate_pair(w / jn, ev[0], ei[0]);
      }
      if (!jac_sync(ctl, ++nbar * G, &s_ok)) return;
      double *const done = An;
      An = A;
      A = done;
    }
  }
  for (int i = gt; i < r; i += gn) eval[i] = __ldcg(A + i * r + i);
  if (gt == 0) ctl->sweeps = sweep;
}

// Column c of L^-1 by forward substitution in one warp, rows lane + 32 t in
// z[t] (r <= 32 RL): x_k = z_k / l_kk goes round by shuffles, then z_i -= l_ik x_k
// below.  Two FP64 operations and a shuffle deep a step; column k of L (a row of
// LT) is requested four steps ahead.
template <int RL>
__device__ void chol_inv_column(int c, int r, const double *LT, const double *inv, int lane, double (&z)[RL]) {
#pragma unroll
  for (int t = 0; t < RL; ++t) z[t] = lane + 32 * t == c ? 1.0 : 0.0;
  double ring[4][RL];
  auto request = [&](int k, double (&v)[RL]) {
#pragma unroll
    for (int t = 0; t < RL; ++t) {
      const int i = lane + 32 * t;
      v[t] = (k < r && i < r && i > k) ? __ldcg(LT + k * r + i) : 0.0;
    }
  };
  const int k0 = c & ~3;  // the steps before c find zeros
#pragma unroll
  for (int g = 0; g < 4; ++g) request(k0 + g, ring[g]);
#pragma unroll
  for (int t = 0; t < RL; ++t) {
    if (32 * t + 31 < k0 || 32 * t >= r) continue;
    for (int kb = max(32 * t, k0); kb < min(32 * t + 32, r); kb += 4) {
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int k = kb + g;
        if (k < r) {
          const double x = __shfl_sync(0xffffffffu, z[t], k & 31) * inv[k];
          if (lane == (k & 31)) z[t] = x;
#pragma unroll
          for (int u = t; u < RL; ++u)
            if (32 * u < r) z[u] = fma(-ring[g][u], x, z[u]);  // zero at and above row k
        }
        request(k + 4, ring[g]);
      }
    }
  }
}

// Cholesky factor and inverse of a symmetric positive definite r x r FP64
// matrix A (overwritten), r <= kMaxRitz: A = L L^T in panels of 32 columns, then
// X = L^-1 column by column.  Per panel every block factors the 32 x 32
// diagonal block for itself, warps solve the rows below it, a grid barrier, then
// the trailing entries take the panel's 32 terms, and another: 2 r/32 grid
// barriers where one per column took 2 r.  The columns of X are independent: a
// warp each, no barrier.
// What bounds it is the chain of FP64 operations, 64 cycles each a warp and SM
// quarter (a division or square root 430 to 680).  The diagonal block runs in
// four warps, one a quarter, lane = row, every fourth column a warp: a step is
// the pivot's reciprocal (FP32 and one third-order step), the scaled column, and
// the next pivot's column, which its warp publishes before the other columns
// take the step; the columns are scaled by 1/sqrt at the end, side by side.
// 1185 -> 287 us at r = 216, 345 -> 85 us at r = 66 (19 us of each whole panel).
// L (lower, zeros above) and LT (its transpose, scratch) are required; Linv,
// LinvT64 = L^-T and LinvT32 (FP32) are written when given.  status: 1 if a
// pivot was not positive (it is taken as 1), 2 if a grid barrier expired.  *ill,
// when given: set to 1 if the diagonal of L spans more than 1e5.
constexpr int kCholNb = 32;
__global__ void __launch_bounds__(kJacThreads) k_chol_inv(double *__restrict__ A, int r, double *__restrict__ L,
                                                         double *__restrict__ LT, double *Linv, double *LinvT64,
                                                         float *LinvT32, int *status, int *ill, JacCtl *ctl) {
  __shared__ double Dc[kCholNb][kCholNb + 1], inv[kMaxRitz];  // the diagonal block by columns: Dc[k][i]
  __shared__ int s_ok;
  const int G = gridDim.x, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, w = tid >> 5;
  const int gt = blockIdx.x * nt + tid, gn = G * nt, rr = r * r;
  unsigned nbar = 0;
  for (int e = gt; e < rr; e += gn)
    if (e % r > e / r) L[e] = 0.0;
  for (int j0 = 0; j0 < r; j0 += kCholNb) {
    const int jb = min(kCholNb, r - j0), j1 = j0 + jb;
    // the lower half; past the matrix the identity, so that a short panel runs alike
    for (int e = tid; e < kCholNb * kCholNb; e += nt) {
      const int i = e >> 5, k = e & 31;
      if (k <= i) Dc[k][i] = i < jb ? __ldcg(A + (j0 + i) * r + j0 + k) : (i == k ? 1.0 : 0.0);
    }
    __syncthreads();
    if (w < 4) {
      double a[8];  // column w + 4 u, row lane (u counted from the current pivot's group)
#pragma unroll
      for (int u = 0; u < 8; ++u) a[u] = w + 4 * u <= lane ? Dc[w + 4 * u][lane] : 0.0;
      for (int jg = 0; jg < jb; jg += 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int j = jg + q;
          // column j is final in Dc
          const double v = lane >= j ? Dc[j][lane] : 0.0;
          double d = Dc[j][j];
          const int hd = __double2hiint(d);  // positive, not NaN: an integer test
          if (!((hd > 0 && hd <= 0x7ff00000) || (hd == 0 && __double2loint(d) != 0))) {
            if (gt == 0 && j < jb) atomicMax(status, 1);
            d = 1.0;
          }
          const double g = -(v * recip64(d));
          // the next pivot's column first, published at once
          const int nw = (q + 1) & 3, nu = q == 3 ? 1 : 0;
          if (w == nw && j + 1 < kCholNb) {
            a[nu] = fma(g, Dc[j][j + 1], a[nu]);
            if (lane > j) Dc[j + 1][lane] = a[nu];
          }
          asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int k = jg + w + 4 * u;
            if (k > j + 1 && k < kCholNb) a[u] = fma(g, Dc[j][k], a[u]);
          }
        }
#pragma unroll
        for (int u = 0; u < 7; ++u) a[u] = a[u + 1];
      }
    }
    __syncthreads();
    if (tid < jb) {
      const double d = Dc[tid][tid];
      const double q = rsqrt(d > 0.0 ? d : 1.0);
      inv[j0 + tid] = q;
    }
    __syncthreads();
    for (int e = tid; e < jb * jb; e += nt) {
      const int k = e / jb, i = e % jb;
      if (k <= i) {
        double x = Dc[k][i];
        if (k == i && !(x > 0.0)) x = 1.0;
        Dc[k][i] = x * inv[j0 + k];
      }
    }
    __syncthreads();
    if (blockIdx.x == 0)
      for (int e = tid; e < jb * jb; e += nt) {
        const int k = e / jb, i = e % jb;
        if (k <= i) {
          L[(j0 + i) * r + j0 + k] = Dc[k][i];
          LT[(j0 + k) * r + j0 + i] = Dc[k][i];
        }
      }
    // rows below: x L11^T = a, lane k holds column k
    for (int i = j1 + (gt >> 5); i < r; i += gn >> 5) {
      double a = lane < jb ? __ldcg(A + i * r + j0 + lane) : 0.0;
      for (int k = 0; k < jb; ++k) {
        const double x = __shfl_sync(0xffffffffu, a, k) * inv[j0 + k];
        if (lane == k) a = x;
        else if (lane > k && lane < jb) a = fma(-x, Dc[k][lane], a);
      }
      if (lane < jb) {
        L[i * r + j0 + lane] = a;
        LT[(j0 + lane) * r + i] = a;
      }
    }
    if (!jac_sync(ctl, ++nbar * G, &s_ok)) {
      if (tid == 0) atomicMax(status, 2);
      return;
    }
    if (j1 >= r) break;
    const int m = r - j1;
    for (int e = gt; e < m * m; e += gn) {
      const int i = j1 + e / m, k = j1 + e % m;
      if (k > i) continue;
      double v = __ldcg(A + i * r + k);
#pragma unroll 8
      for (int q = 0; q < kCholNb; ++q)  // a panel with columns after it is whole
        v = fma(-__ldcg(LT + (j0 + q) * r + i), __ldcg(LT + (j0 + q) * r + k), v);
      A[i * r + k] = v;
    }
    if (!jac_sync(ctl, ++nbar * G, &s_ok)) {
      if (tid == 0) atomicMax(status, 2);
      return;
    }
  }
  if (ill && blockIdx.x == 0 && w == 0) {  // every block has the whole of inv
    double mn = inv[0], mx = inv[0];
    bool num = true;
    for (int i = lane; i < r; i += 32) {
      const double v = inv[i];
      num = num && v > 0.0;
      mn = fmin(mn, v);
      mx = fmax(mx, v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    num = __all_sync(0xffffffffu, num);
    if (lane == 0 && !(num && mx <= 1e5 * mn)) *ill = 1;
  }
  if (!Linv && !LinvT64 && !LinvT32) return;
  // warp w of block b takes columns b + G w, b + G (w + 8), ...: one a quarter first
  auto columns = [&](auto rl) {
    constexpr int RL = decltype(rl)::value;
    for (int c = blockIdx.x + G * w; c < r; c += G * (nt >> 5)) {
      double z[RL];
      chol_inv_column<RL>(c, r, LT, inv, lane, z);
#pragma unroll
      for (int t = 0; t < RL; ++t) {
        const int i = lane + 32 * t;
        if (i >= r) continue;
        const double x = c <= i ? z[t] : 0.0;
        if (Linv) Linv[i * r + c] = x;
        if (LinvT64) LinvT64[c * r + i] = x;
        if (LinvT32) LinvT32[c * r + i] = (float)x;
      }
    }
  };
  if (r <= 128) columns(std::integral_constant<int, 4>());
  else if (r <= 256) columns(std::integral_constant<int, 8>());
  else if (r <= 512) columns(std::integral_constant<int, 16>());
  else columns(std::integral_constant<int, (kMaxRitz + 31) / 32>());
}

// B = C1 C2^-1 for r x r FP64 matrices (C2 general, row-major): Gauss-Jordan
// elimination with partial pivoting (largest |pivot| among the rows not yet
// used, lowest index on ties) of C2^T B^T = C1^T, spread over the grid, one
// grid barrier per column.  M and R are r x r scratch (the system and its
// right-hand sides, eliminated in place; column j of M is left as it was once
// eliminated, being read no more).  status: 1 if a pivot is zero (C2
// singular), 2 if a grid barrier expired.
__global__ void __launch_bounds__(kJacThreads) k_solve_right(const double *__restrict__ C1,
                                                            const double *__restrict__ C2, int r,
                                                            double *__restrict__ M, double *__restrict__ R,
                                                            double *__restrict__ B, int *status, JacCtl *ctl) {
  __shared__ unsigned char used[kMaxDim];
  __shared__ int piv[kMaxDim];
  __shared__ unsigned long long red_v[kJacThreads / 32];
  __shared__ int red_i[kJacThreads / 32];
  __shared__ int s_ok, s_p;
  const int G = gridDim.x, tid = threadIdx.x, nt = blockDim.x;
  const int gt = blockIdx.x * nt + tid, gn = G * nt, rr = r * r;
  unsigned nbar = 0;
  for (int e = gt; e < rr; e += gn) {
    const int i = e / r, c = e % r;
    M[e] = C2[c * r + i];
    R[e] = C1[c * r + i];
  }
  for (int i = tid; i < r; i += nt) used[i] = 0;
  if (!jac_sync(ctl, ++nbar * G, &s_ok)) {
    if (tid == 0) atomicMax(status, 2);
    return;
  }
  for (int j = 0; j < r; ++j) {
    // largest |pivot|, lowest row on ties, as one key: magnitudes compare as
    // their bits (integer units; an FP64 comparison takes 64 cycles), NaN is
    // no candidate
    unsigned long long bv = 0;  // bits + 1
    int bi = r;
    for (int i = tid; i < r; i += nt)
      if (!used[i]) {
        const unsigned long long v = (unsigned long long)__double_as_longlong(__ldcg(M + i * r + j)) & 0x7fffffffffffffffull;
        if (v <= 0x7ff0000000000000ull && v + 1 > bv) {
          bv = v + 1;
          bi = i;
        }
      }
    for (int m = 16; m > 0; m >>= 1) {
      const unsigned long long ov = __shfl_xor_sync(0xffffffffu, bv, m);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, m);
      if (ov > bv || (ov == bv && oi < bi)) {
        bv = ov;
        bi = oi;
      }
    }
    if ((tid & 31) == 0) {
      red_v[tid >> 5] = bv;
      red_i[tid >> 5] = bi;
    }
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < nt / 32; ++w)
        if (red_v[w] > bv || (red_v[w] == bv && red_i[w] < bi)) {
          bv = red_v[w];
          bi = red_i[w];
        }
      if (bv <= 1) {  // zero, or no finite candidate
        if (blockIdx.x == 0) atomicMax(status, 1);
        if (bi >= r)  // no finite candidate: take the first unused row
          for (bi = 0; bi < r && used[bi]; ++bi) {
          }
      }
      used[bi] = 1;
      piv[j] = bi;
      s_p = bi;
    }
    __syncthreads();
    const int p = s_p;
    const double mpj = __ldcg(M + p * r + j);
    const double inv = mpj != 0.0 ? 1.0 / mpj : 0.0;
    const int wm = r - j - 1, width = wm + r;  // columns j+1 .. r-1 of M, then every column of R
    for (int e = gt; e < r * width; e += gn) {
      const int i = e / width, c = e % width;
      if (i == p) continue;
      const double f = __ldcg(M + i * r + j) * inv;
      if (c < wm) {
        const int cc = j + 1 + c;
        M[i * r + cc] = __ldcg(M + i * r + cc) - f * __ldcg(M + p * r + cc);
      } else {
        const int cc = c - wm;
        R[i * r + cc] = __ldcg(R + i * r + cc) - f * __ldcg(R + p * r + cc);
      }
    }
    if (!jac_sync(ctl, ++nbar * G, &s_ok)) {
      if (tid == 0) atomicMax(status, 2);
      return;
    }
  }
  // row j of B^T is the pivot row of column j, divided by its pivot
  for (int e = gt; e < rr; e += gn) {
    const int j = e / r, c = e % r, p = piv[j];
    const double d = __ldcg(M + p * r + j);
    B[c * r + j] = d != 0.0 ? __ldcg(R + p * r + c) / d : 0.0;
  }
}

// Z = sP * Z - a0 * M1 (M1^T Q)  (rank-one part of M2 applied to Q), r columns.
__global__ void k_rank1_fix(double *Z, const double *M1, const double *m1q, int V, int r, double sP, double a0) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)V * r) return;
  const int i = (int)(e / r), j = (int)(e % r);
  Z[e] = sP * Z[e] - a0 * M1[i] * m1q[j];
}

// Per column of U (V x D) and slab of rows (blockIdx.y), the entry of largest
// magnitude: |u| and row (the lowest on ties) in a key per slab.  One block per
// 32 columns, whole rows read.
__global__ void __launch_bounds__(256) k_col_peak(const double *U, int V, int D, int slab, double *pv, int *pi) {
  __shared__ double bv[8][33];
  __shared__ int bi[8][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  const int r0 = blockIdx.y * slab, r1 = min(V, r0 + slab);
  double best = -1.0;
  int at = 0x7fffffff;
  if (c < D) {
#pragma unroll 4
    for (int m = r0 + w; m < r1; m += 8) {  // rows ascend: the first of equals stays
      const double a = fabs(U[(long long)m * D + c]);
      if (a > best) {
        best = a;
        at = m;
      }
    }
  }
  bv[w][lane] = best;
  bi[w][lane] = at;
  __syncthreads();
  if (w == 0 && c < D) {
#pragma unroll
    for (int q = 1; q < 8; ++q)
      if (bv[q][lane] > best || (bv[q][lane] == best && bi[q][lane] < at)) {
        best = bv[q][lane];
        at = bi[q][lane];
      }
    pv[blockIdx.y * D + c] = best;
    pi[blockIdx.y * D + c] = at;
  }
}

// W = U_D Lambda^-1/2 with the sign of each eigenvector fixed so that its
// largest-magnitude entry is positive (lowest index on ties), and m1 += W^T M1
// over the block's rows (m1_64 zeroed before).  Blocks as k_col_peak's, whose
// nslab peaks each block folds for its columns.
__global__ void __launch_bounds__(256) k_make_w(const double *U, int V, int D, int slab, const double *pv, const int *pi,
                                                int nslab, const double *lam, const double *M1, float *W32,
                                                double *m1_64) {
  __shared__ double red[8][33], scale[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  const int r0 = blockIdx.y * slab, r1 = min(V, r0 + slab);
  if (w == 0 && c < D) {
    double best = -1.0;
    int at = 0x7fffffff;
    for (int q = 0; q < nslab; ++q) {
      const double a = pv[q * D + c];
      if (a > best) {  // slabs ascend in rows
        best = a;
        at = pi[q * D + c];
      }
    }
    if (at >= V) at = 0;  // every entry NaN
    scale[lane] = (U[(long long)at * D + c] < 0 ? -1.0 : 1.0) / sqrt(lam[c]);
  }
  __syncthreads();
  double s = 0.0;
  if (c < D) {
    const double sc = scale[lane];
#pragma unroll 4
    for (int m = r0 + w; m < r1; m += 8) {
      const float x = (float)(U[(long long)m * D + c] * sc);
      W32[(long long)m * D + c] = x;
      s = fma((double)x, M1[m], s);
    }
  }
  red[w][lane] = s;
  __syncthreads();
  if (w == 0 && c < D) {
#pragma unroll
    for (int q = 1; q < 8; ++q) s += red[q][lane];
    atomicAdd(m1_64 + c, s);
  }
}

__global__ void k_m1_f32(const double *m1_64, int D, int Dp, float *m1) {
  const int i = threadIdx.x + blockIdx.x * blockDim.x;
  if (i < Dp) m1[i] = i < D ? (float)m1_64[i] : 0.f;
}

// Enqueues W, m1 and U of a whitening from U64 (V x D) and lam; peaks: kWSlabs x
// D doubles and as many ints, m1_64: D.
constexpr int kWSlabs = 64;
void make_whitening(tlda_ctx *ctx, const double *U64, const double *lam, const double *M1, double *pv, int *pi,
                    double *m1_64, cudaStream_t s) {
  const int V = ctx->V, D = ctx->D, slab = std::max(8, (V + kWSlabs - 1) / kWSlabs), ns = (V + slab - 1) / slab;
  const dim3 g((D + 31) / 32, ns);
  cudaMemsetAsync(m1_64, 0, sizeof(double) * D, s);
  k_col_peak<<<g, 256, 0, s>>>(U64, V, D, slab, pv, pi);
  k_make_w<<<g, 256, 0, s>>>(U64, V, D, slab, pv, pi, ns, lam, M1, ctx->W32, m1_64);
  k_m1_f32<<<1, kMaxDim, 0, s>>>(m1_64, D, ctx->Dp, ctx->m1);
  launch_make_u(ctx->W32, ctx->m1, V, D, ctx->Dp, ctx->U32, ctx->U16, s);
}

// ------------------------------------------------------------------ unwhitening
// n2_i = ||phi_i||^2 and alpha_i ~ ||phi_i||^-6, normalised (one block).
__global__ void __launch_bounds__(kMaxDim) k_unwhiten_norms(const float *Phi, int D, int K, double *n2_out, double *alpha) {
  __shared__ double red[kMaxDim];
  const int i = threadIdx.x;
  double a = 0.0;
  if (i < K) {
    double n2 = 0.0;
#pragma unroll 8
    for (int j = 0; j < D; ++j) {
      const double p = (double)Phi[j * K + i];
      n2 = fma(p, p, n2);
    }
    n2_out[i] = n2;
    a = pow(n2, -3.0);
  }
  red[i] = a;
  __syncthreads();
  for (int w = kMaxDim / 2; w > 0; w >>= 1) {
    if (i < w) red[i] += red[i + w];
    __syncthreads();
  }
  if (i < K) alpha[i] = a / red[0];
}

// Column sums of max(mu, 0) (V x K) into sum (zeroed before): one block per 32
// columns and slab of rows; then mu = max(mu, 0) / sum (1 where that is 0).
// Both read whole rows (a block per column would touch a 32-byte sector for
// each entry).
__global__ void __launch_bounds__(256) k_clip_sum(const double *mu, int V, int K, int slab, double *sum) {
  __shared__ double red[8][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  const int r0 = blockIdx.y * slab, r1 = min(V, r0 + slab);
  double v = 0.0;
  if (c < K) {
#pragma unroll 4
    for (int r = r0 + w; r < r1; r += 8) {
      const double x = mu[(long long)r * K + c];
      v += x > 0.0 ? x : 0.0;
    }
  }
  red[w][lane] = v;
  __syncthreads();
  if (w == 0 && c < K) {
#pragma unroll
    for (int q = 1; q < 8; ++q) v += red[q][lane];
    atomicAdd(sum + c, v);
  }
}

__global__ void __launch_bounds__(256) k_clip_scale(double *mu, int V, int K, int slab, const double *sum) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  const int r0 = blockIdx.y * slab, r1 = min(V, r0 + slab);
  if (c >= K) return;
  const double z = sum[c] > 0.0 ? sum[c] : 1.0, inv = 1.0 / z;
#pragma unroll 4
  for (int r = r0 + w; r < r1; r += 8) {
    const double v = mu[(long long)r * K + c], x = v > 0.0 ? v : 0.0, q = x * inv;
    mu[(long long)r * K + c] = fma(fma(-z, q, x), inv, q);  // x / z to rounding, without a division an entry
  }
}

tlda_status fail(tlda_ctx *c, tlda_status s, const char *msg) {
  if (c) c->err = msg;
  return s;
}

#define CKF(call)                                                                                 \
  do {                                                                                            \
    cudaError_t e_ = (call);                                                                      \
    if (e_ != cudaSuccess) {                                                                      \
      ctx->err = std::string(#call) + ": " + cudaGetErrorString(e_);                              \
      return e_ == cudaErrorMemoryAllocation ? TLDA_ERR_OOM : TLDA_ERR_CUDA;                      \
    }                                                                                             \
  } while (0)

template <class T>
void dfree(T *&p) {
  if (p) cudaFree(p);
  p = nullptr;
}

template <class T>
cudaError_t dalloc(T **p, size_t n, bool zero = false) {
  if (n == 0) n = 1;
  cudaError_t e = cudaMalloc(reinterpret_cast<void **>(p), n * sizeof(T));
  if (e == cudaSuccess && zero) e = cudaMemset(*p, 0, n * sizeof(T));
  return e;
}

// Arrays laid out one after the other (256-byte aligned); base null: only measured.
struct Carver {
  char *base;
  size_t off = 0;
  template <class T>
  void take(T *&p, size_t n) {
    off = (off + 255) & ~size_t(255);
    p = base ? reinterpret_cast<T *>(base + off) : nullptr;
    off += n * sizeof(T);
  }
};

// Scratch of a FINALIZE: one allocation (each cudaMalloc and
// cudaFree takes the host some 15 us), freed on every exit path.
struct Scratch {
  void *ptr = nullptr;
  template <class F>
  cudaError_t carve(F lay) {
    Carver m{nullptr};
    lay(m);
    const cudaError_t e = cudaMalloc(&ptr, m.off);
    if (e != cudaSuccess) {
      ptr = nullptr;
      return e;
    }
    Carver c{static_cast<char *>(ptr)};
    lay(c);
    return cudaSuccess;
  }
  ~Scratch() {
    if (ptr) cudaFree(ptr);
  }
};

// Blocks of the grid-wide Jacobi, Cholesky and solve kernels: one per SM, all
// co-resident (cooperative launch).
int coop_grid() {
  static int g = -1;
  if (g >= 0) return g;
  int dev = 0, sms = 0, coop = 0, pj = 0, pc = 0, ps = 0;
  g = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return g;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (!coop || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pj, k_jacobi, kJacThreads, 0) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pc, k_chol_inv, kJacThreads, 0) != cudaSuccess || pj < 1 ||
      pc < 1 || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, k_solve_right, kJacThreads, 0) != cudaSuccess ||
      ps < 1)
    return g;
  g = std::min(sms, kJacMaxGrid);
  return g;
}

// The context's control block for those kernels, zeroed on its stream.
tlda_status coop_ctl(tlda_ctx *ctx, JacCtl **out, cudaStream_t s) {
  if (coop_grid() < 1) return fail(ctx, TLDA_ERR_CUDA, "cooperative launch unavailable for the dense FP64 kernels");
  if (!ctx->coop_ctl) CKF(cudaMalloc(&ctx->coop_ctl, sizeof(JacCtl)));
  CKF(cudaMemsetAsync(ctx->coop_ctl, 0, sizeof(JacCtl), s));
  *out = static_cast<JacCtl *>(ctx->coop_ctl);
  return TLDA_OK;
}

// The context's exponents for the FP64 products.
tlda_status g64_exps(tlda_ctx *ctx, int **out) {
  if (!ctx->g64_exp) CKF(dalloc(&ctx->g64_exp, 2 * (size_t)ctx->V + 2 * kExpCols));
  *out = ctx->g64_exp;
  return TLDA_OK;
}

// Diagonalises the symmetric r x r matrix A (device, overwritten, as is the r x r
// scratch): eigenvalues to ev, eigenvector rows to Et.  Synchronises.
tlda_status run_jacobi(tlda_ctx *ctx, double *A, double *scratch, int r, double *Et, double *ev, cudaStream_t s) {
  if (r > kMaxRitz) return fail(ctx, TLDA_ERR_INVALID, "eigenproblem above the solver's order");
  JacCtl *ctl = nullptr;
  if (tlda_status st = coop_ctl(ctx, &ctl, s)) return st;
  int ms = 40;
  void *args[] = {&A, &scratch, &r, &Et, &ev, &ms, &ctl};
  CKF(cudaLaunchCooperativeKernel((const void *)k_jacobi, dim3(coop_grid()), dim3(kJacThreads), args, 0, s));
  int hs[3];
  CKF(cudaMemcpyAsync(hs, &ctl->bar, sizeof hs, cudaMemcpyDeviceToHost, s));
  CKF(cudaStreamSynchronize(s));
  if (hs[1]) return fail(ctx, TLDA_ERR_TIMEOUT, "grid barrier of the Jacobi eigensolver expired");
  ctx->jacobi_sweeps = hs[2];
  return TLDA_OK;
}

// Enqueues k_chol_inv (asynchronous; failures land in *status).
tlda_status run_chol_inv(tlda_ctx *ctx, double *A, int r, double *L, double *Z, double *Linv, double *LinvT64,
                         float *LinvT32, int *status, cudaStream_t s, int *ill = nullptr) {
  if (r > kMaxRitz) return fail(ctx, TLDA_ERR_INVALID, "matrix above the Cholesky kernel's order");
  JacCtl *ctl = nullptr;
  if (tlda_status st = coop_ctl(ctx, &ctl, s)) return st;
  void *args[] = {&A, &r, &L, &Z, &Linv, &LinvT64, &LinvT32, &status, &ill, &ctl};
  CKF(cudaLaunchCooperativeKernel((const void *)k_chol_inv, dim3(coop_grid()), dim3(kJacThreads), args, 0, s));
  return TLDA_OK;
}

// Enqueues k_solve_right: B = C1 C2^-1 (asynchronous; failures land in *status).
tlda_status run_solve_right(tlda_ctx *ctx, const double *C1, const double *C2, int r, double *M, double *R,
                            double *B, int *status, cudaStream_t s) {
  JacCtl *ctl = nullptr;
  if (tlda_status st = coop_ctl(ctx, &ctl, s)) return st;
  void *args[] = {&C1, &C2, &r, &M, &R, &B, &status, &ctl};
  CKF(cudaLaunchCooperativeKernel((const void *)k_solve_right, dim3(coop_grid()), dim3(kJacThreads), args, 0, s));
  return TLDA_OK;
}

// Maps the status word of k_chol_inv / k_solve_right to the call's result.
tlda_status chol_status(tlda_ctx *ctx, int st, const char *breakdown) {
  if (st >= 2) return fail(ctx, TLDA_ERR_TIMEOUT, "grid barrier of a dense FP64 kernel expired");
  if (st == 1) return fail(ctx, TLDA_ERR_NUMERIC, breakdown);
  return TLDA_OK;
}

tlda_status finalize(tlda_ctx *ctx) {
  cudaStream_t s = ctx->stream;
  const int V = ctx->V, D = ctx->D;
  int r = round_up(D + kOversample, 2);
  if (r > V) r = V - (V & 1);
  if (r < D) return fail(ctx, TLDA_ERR_INVALID, "vocabulary too small for the whitening dimension");
  unsigned long long TS[3];
  int ferr = 0;
  CKF(cudaMemcpyAsync(TS, ctx->TS, sizeof TS, cudaMemcpyDeviceToHost, s));
  CKF(cudaMemcpyAsync(&ferr, ctx->fit_err, sizeof ferr, cudaMemcpyDeviceToHost, s));
  CKF(cudaStreamSynchronize(s));
  if (ferr) return fail(ctx, TLDA_ERR_INVALID, "corrupt CSR chunk in fit_moments");
  if (TS[0] == 0 || TS[1] == 0) return fail(ctx, TLDA_ERR_NUMERIC, "no token pairs accumulated");
  const double a0 = ctx->p.alpha0, sP = (a0 + 1.0) / (double)TS[1];
  const long long VV = (long long)V * V;
  int *ex = nullptr;
  if (tlda_status st = g64_exps(ctx, &ex)) return st;
  const int sms = ctx->num_sms, splits = sgemm_splits(V, r, V, sms);
  // one allocation, freed on every exit path
  double *M1 = nullptr, *Q64 = nullptr, *Z64 = nullptr, *G = nullptr, *Linv = nullptr, *LinvT64 = nullptr;
  double *Zr = nullptr, *Pv = nullptr;
  int *Pi = nullptr;
  double *Bm = nullptr, *Ev = nullptr, *ev = nullptr, *m1q = nullptr, *U64 = nullptr, *lam = nullptr, *Ek = nullptr;
  float *M2 = nullptr, *Om = nullptr, *Y = nullptr, *Qf = nullptr, *LinvT32 = nullptr, *part = nullptr;
  int *status = nullptr;
  Scratch sc;
  const size_t Vr = (size_t)V * r, r2 = (size_t)r * r;
  CKF(sc.carve([&](Carver &c) {
    c.take(M1, V);
    c.take(Q64, Vr);
    c.take(Z64, Vr);
    c.take(G, r2);
    c.take(Linv, r2);
    c.take(LinvT64, r2);
    c.take(Zr, r2);
    c.take(Bm, r2);
    c.take(Ev, r2);
    c.take(ev, r);
    c.take(Ek, (size_t)r * D);
    c.take(m1q, r);
    c.take(U64, (size_t)V * D);
    c.take(lam, D);
    c.take(Pv, (size_t)kWSlabs * D);
    c.take(Pi, (size_t)kWSlabs * D);
    c.take(M2, (size_t)VV);
    c.take(Om, Vr);
    c.take(Y, Vr);
    c.take(Qf, Vr);
    c.take(LinvT32, r2);
    c.take(part, splits > 1 ? splits * Vr : 1);
    c.take(status, 2);
  }));
  k_m1<<<(V + 255) / 256, 256, 0, s>>>(ctx->Ccnt, ctx->TS, V, M1);
  k_m2_mirror<<<dim3((V + 31) / 32, (V + 31) / 32), 256, 0, s>>>(ctx->P64, M1, V, sP, a0, M2);
  k_gauss<<<(unsigned)(((long long)V * r + 255) / 256), 256, 0, s>>>(Om, (long long)V * r, ctx->p.seed * 0x100000001B3ull + 17);
  // one CholeskyQR pass: out = in L^-T with L L^T = in^T in (FP64 Gram)
  auto cholqr_pass = [&](const float *in, float *out) -> tlda_status {
    gemm_tn64(in, r, in, r, G, r, r, r, V, ex, V, sms, s);
    if (tlda_status st = run_chol_inv(ctx, G, r, Linv, Zr, nullptr, nullptr, LinvT32, status, s, status + 1)) return st;
    sgemm(in, r, LinvT32, r, out, V, r, r, nullptr, 1, s);
    return TLDA_OK;
  };
  // Y = M2 Q, then CholeskyQR.  A single pass keeps the same span, and the columns
  // orthonormal to the FP32 rounding of Q times the condition of Y.  While that is
  // small the next product needs no more, and a second pass is taken at the end
  // only; where a factor's diagonal spans more than 1e5 (a spectrum that falls by
  // as much within r columns) the loss would grow from product to product until
  // the factor breaks down, and the iteration starts over with two passes each.
  const int n_iter = 24;
  auto iterate = [&](int passes) -> tlda_status {
    CKF(cudaMemsetAsync(status, 0, 2 * sizeof(int), s));
    for (int it = 0; it <= n_iter; ++it) {
      sgemm(M2, V, it ? Qf : Om, r, Y, V, r, V, part, splits, s);
      if (tlda_status st = cholqr_pass(Y, Qf)) return st;
      if (passes == 2) {
        if (tlda_status st = cholqr_pass(Qf, Y)) return st;
        std::swap(Qf, Y);
      }
    }
    return TLDA_OK;
  };
  int hstat[2];
  for (int passes = 1; passes <= 2; ++passes) {
    if (tlda_status st = iterate(passes)) return st;
    CKF(cudaMemcpyAsync(hstat, status, sizeof hstat, cudaMemcpyDeviceToHost, s));
    CKF(cudaStreamSynchronize(s));
    if (!hstat[1] && hstat[0] != 1) break;
  }
  if (tlda_status st = chol_status(ctx, hstat[0], "subspace basis lost rank (CholeskyQR breakdown)")) return st;
  // FP64 Rayleigh-Ritz on the exact M2 = sP P - a0 M1 M1^T
  // one FP64 CholeskyQR pass makes Q64 orthonormal to FP64 accuracy
  gemm_tn64(Qf, r, Qf, r, G, r, r, r, V, ex, V, sms, s);
  if (tlda_status st = run_chol_inv(ctx, G, r, Linv, Zr, nullptr, LinvT64, nullptr, status, s)) return st;
  gemm_nn64(Qf, r, LinvT64, r, Q64, r, V, r, r, ex, V, sms, s);
  gemm_nn64(ctx->P64, V, Q64, r, Z64, r, V, r, V, ex, V, sms, s);
  vec_tn64(M1, Q64, V, r, m1q, s);
  k_rank1_fix<<<(unsigned)(((long long)V * r + 255) / 256), 256, 0, s>>>(Z64, M1, m1q, V, r, sP, a0);
  gemm_tn64(Q64, r, Z64, r, Bm, r, r, r, V, ex, V, sms, s);
  CKF(cudaGetLastError());
  if (tlda_status js = run_jacobi(ctx, Bm, G, r, Ev, ev, s)) return js;
  std::vector<double> hev(r), hEv((size_t)r * r);
  CKF(cudaMemcpyAsync(hev.data(), ev, sizeof(double) * r, cudaMemcpyDeviceToHost, s));
  CKF(cudaMemcpyAsync(hEv.data(), Ev, sizeof(double) * r * r, cudaMemcpyDeviceToHost, s));
  CKF(cudaMemcpyAsync(hstat, status, sizeof hstat, cudaMemcpyDeviceToHost, s));
  CKF(cudaStreamSynchronize(s));
  if (tlda_status st = chol_status(ctx, hstat[0], "subspace basis lost rank (CholeskyQR breakdown)")) return st;
  // order the Ritz pairs by descending value and keep D of them
  std::vector<int> ord(r);
  for (int i = 0; i < r; ++i) ord[i] = i;
  std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return hev[x] > hev[y]; });
  std::vector<double> hEk((size_t)r * D), hlam(D);
  for (int j = 0; j < D; ++j) {
    hlam[j] = hev[ord[j]];
    for (int i = 0; i < r; ++i) hEk[(size_t)i * D + j] = hEv[(size_t)ord[j] * r + i];
  }
  if (!(hlam[D - 1] > 1e-12 * hlam[0]))
    return fail(ctx, TLDA_ERR_NUMERIC, "M2 has fewer than D positive eigenvalues");
  CKF(cudaMemcpyAsync(Ek, hEk.data(), sizeof(double) * r * D, cudaMemcpyHostToDevice, s));
  CKF(cudaMemcpyAsync(lam, hlam.data(), sizeof(double) * D, cudaMemcpyHostToDevice, s));
  gemm_nn64(Q64, r, Ek, D, U64, D, V, D, r, ex, V, sms, s);
  make_whitening(ctx, U64, lam, M1, Pv, Pi, m1q, s);
  CKF(cudaGetLastError());
  CKF(cudaStreamSynchronize(s));
  ctx->eig = hlam;
  ctx->whitened = true;
  ctx->fitted = true;
  return TLDA_OK;
}

// ------------------------------------------------------------------ fully online mode
// The sketch Z = P Omega of the pair counts P = sum_d (f_d f_d^T - diag f_d),
// taken over a piece of documents at a time as
//   Z += F^T S - diag(c) Omega,   S = F Omega,   c = F^T 1,
// with F the piece's document x word counts.  Row m of F^T S sums f_dm s_d
// over the documents holding word m, which needs the piece's nonzeros grouped
// by word (its transpose).  Per piece:
//   k_sk_rows     one warp per document: validation, the token statistics,
//                 s_d = f_d^T Omega into row d of S, and the number of
//                 nonzeros of each word;
//   scan          those numbers become each word's first slot;
//   k_sk_scatter  one warp per document: each nonzero (document, count) into
//                 a slot of its word;
//   k_sk_z        one warp per run of kSkRun consecutive slots: for each word
//                 met, the run's part of sum_d f_dm (s_d - Omega_m) added to
//                 Z_m and sum_d f_dm to C_m; plainly when all the word's
//                 slots lie in the run, with FP64 atomics when they cross its
//                 ends.
// Precision: the products and the sums within a document (s_d) and within a
// run (at most kSkRun terms) are FP32, from an FP32 copy of Omega; Z
// accumulates the runs in FP64.  (GB300's FP64 rate is 1/64 of its FP32
// rate: with FP64 products the sketch would be bound by them.)
// The per-nonzero work is two row gathers (Omega_m, then s_d) and no atomics
// on Z.  The slots of a word are filled in no fixed order, so Z is not
// bitwise reproducible (its sums are reordered).  A document that fails
// validation adds nothing and sets *err.
constexpr int kSkPieceDocs = 262144;          // documents per piece (rows of S)
constexpr long long kSkPieceNnz = 16ll << 20;  // nonzeros per piece (slots)
constexpr int kSkRun = 128;                    // slots per warp task of k_sk_z

// Workspace of the sketch (one allocation, made by tlda_online_begin).
struct SketchWs {
  float *S;                          // kSkPieceDocs x r
  int32_t *sd, *sf, *sm;             // slots: document (in the piece), count, word
  int32_t *wcnt, *wfill;             // V + 1 (counts, then first slots), V
  int64_t *scan;                     // scan_blocks(V) + 2
  uint8_t *ok;                       // kSkPieceDocs: the document passed validation
  static size_t al(size_t b) { return (b + 255) & ~size_t(255); }
  static size_t bytes(size_t V, size_t r) {
    return al(sizeof(float) * kSkPieceDocs * r) + 3 * al(sizeof(int32_t) * kSkPieceNnz) +
           al(sizeof(int32_t) * (V + 1)) + al(sizeof(int32_t) * V) + al(sizeof(int64_t) * (scan_blocks((int)V) + 2)) +
           al(kSkPieceDocs);
  }
  SketchWs(void *base, size_t V, size_t r) {
    char *p = static_cast<char *>(base);
    S = reinterpret_cast<float *>(p);
    p += al(sizeof(float) * kSkPieceDocs * r);
    int32_t **slot_bufs[] = {&sd, &sf, &sm};
    for (int32_t **b : slot_bufs) {
      *b = reinterpret_cast<int32_t *>(p);
      p += al(sizeof(int32_t) * kSkPieceNnz);
    }
    wcnt = reinterpret_cast<int32_t *>(p);
    p += al(sizeof(int32_t) * (V + 1));
    wfill = reinterpret_cast<int32_t *>(p);
    p += al(sizeof(int32_t) * V);
    scan = reinterpret_cast<int64_t *>(p);
    p += al(sizeof(int64_t) * (scan_blocks((int)V) + 2));
    ok = reinterpret_cast<uint8_t *>(p);
  }
};

struct SkPiece {
  const int32_t *indptr, *indices, *counts;  // indptr of the piece's first document; absolute offsets
  int n_docs, nz_lo, nz_hi;                  // documents; the piece's offsets lie in [nz_lo, nz_hi]
  int V, r;
};

// The r columns are split over gridDim.y warps per document (or run): block
// row y takes columns y 32 KC + lane + 32 c, KC per lane, so that a warp holds
// few registers and many warps are resident; four rows in flight per warp.
template <int KC>
__global__ void __launch_bounds__(256) k_sk_rows(SkPiece q, const float *__restrict__ Om, float *__restrict__ S,
                                                 int32_t *wcnt, uint8_t *ok, unsigned long long *TS, int *err) {
  const int doc = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (doc >= q.n_docs) return;
  const int p0 = q.indptr[doc], p1 = q.indptr[doc + 1];
  bool bad = p0 < q.nz_lo || p1 > q.nz_hi || p1 < p0;
  long long L = 0;
  if (!bad)
    for (int p = p0 + lane; p < p1; p += 32) {
      const int m = q.indices[p], f = q.counts[p];
      const int prev = p > p0 ? q.indices[p - 1] : -1;
      if (m < 0 || m >= q.V || f <= 0 || m <= prev) bad = true;
      else L += f;
    }
  const bool first = blockIdx.y == 0;  // the column group that also counts
  const int cb = blockIdx.y * 32 * KC;
  if (__any_sync(0xffffffffu, bad)) {
    if (lane == 0 && first) {
      ok[doc] = 0;
      atomicOr(err, 1);
    }
    return;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  float sv[KC];
#pragma unroll
  for (int c = 0; c < KC; ++c) sv[c] = 0.f;
  for (int base = p0; base < p1; base += 32) {
    const int n = min(32, p1 - base);
    const int mj = lane < n ? q.indices[base + lane] : 0, fj = lane < n ? q.counts[base + lane] : 0;
    for (int i = 0; i < n; i += 4) {
      int mm[4];
      float ff[4], row[4][KC];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        mm[u] = __shfl_sync(0xffffffffu, mj, (i + u) & 31);
        ff[u] = (float)__shfl_sync(0xffffffffu, fj, (i + u) & 31);
        if (i + u >= n) ff[u] = 0.f;  // lanes past the end hold word 0, count 0
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < KC; ++c) {
          const int col = cb + lane + 32 * c;
          row[u][c] = col < q.r ? __ldg(Om + (long long)mm[u] * q.r + col) : 0.f;
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < KC; ++c) sv[c] = fmaf(ff[u], row[u][c], sv[c]);
    }
  }
  float *srow = S + (long long)doc * q.r;
#pragma unroll
  for (int c = 0; c < KC; ++c) {
    const int col = cb + lane + 32 * c;
    if (col < q.r) srow[col] = sv[c];
  }
  if (!first) return;
  for (int p = p0 + lane; p < p1; p += 32) atomicAdd(wcnt + q.indices[p] + 1, 1);
  if (lane == 0) {
    ok[doc] = 1;
    if (L > 0) {
      atomicAdd(TS + 0, (unsigned long long)L);
      atomicAdd(TS + 1, (unsigned long long)(L * (L - 1)));
      atomicAdd(TS + 2, (unsigned long long)(L * (L - 1) * (L - 2)));
    }
  }
}

__global__ void __launch_bounds__(256) k_sk_scatter(SkPiece q, const uint8_t *ok, const int32_t *wcnt, int32_t *wfill,
                                                    int32_t *sd, int32_t *sf, int32_t *sm, int *err) {
  const int doc = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (doc >= q.n_docs || !ok[doc]) return;
  const int p0 = q.indptr[doc], p1 = q.indptr[doc + 1];
  for (int p = p0 + lane; p < p1; p += 32) {
    const int m = q.indices[p];
    const long long slot = (long long)wcnt[m] + atomicAdd(wfill + m, 1);
    if (slot < kSkPieceNnz) {  // more slots than the piece's offsets span: overlapping documents
      sd[slot] = doc;
      sf[slot] = q.counts[p];
      sm[slot] = m;
    } else {
      atomicOr(err, 1);
    }
  }
}

template <int KC>
__device__ __forceinline__ void sk_flush(int m, const float (&acc)[KC], long long fs, long long lo, long long hi,
                                         const int32_t *wcnt, int r, int cb, double *Z, unsigned long long *C,
                                         int lane) {
  const bool whole = wcnt[m] >= lo && wcnt[m + 1] <= hi;  // no other run holds word m
  double *z = Z + (long long)m * r;
#pragma unroll
  for (int c = 0; c < KC; ++c) {
    const int col = cb + lane + 32 * c;
    if (col < r) {
      if (whole) z[col] += (double)acc[c];
      else atomicAdd(z + col, (double)acc[c]);
    }
  }
  if (lane == 0 && cb == 0) {
    if (whole) C[m] += (unsigned long long)fs;
    else atomicAdd(C + m, (unsigned long long)fs);
  }
}

template <int KC>
__global__ void __launch_bounds__(256) k_sk_z(const int32_t *__restrict__ wcnt, const int32_t *__restrict__ sd,
                                              const int32_t *__restrict__ sf, const int32_t *__restrict__ sm,
                                              const int64_t *total_p, int r, const float *__restrict__ S,
                                              const float *__restrict__ Om, double *Z, unsigned long long *C,
                                              int *err) {
  const long long total = *total_p;  // valid nonzeros of the piece
  if (total > kSkPieceNnz) {         // k_sk_scatter dropped slots and set *err
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(err, 1);
    return;
  }
  const int lane = threadIdx.x & 31, cb = blockIdx.y * 32 * KC;
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  const long long runs = (total + kSkRun - 1) / kSkRun;
  for (long long t = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < runs; t += nwarps) {
    const long long lo = t * kSkRun, hi = min(total, lo + kSkRun);
    float acc[KC], om[KC];
#pragma unroll
    for (int c = 0; c < KC; ++c) acc[c] = om[c] = 0.f;
    long long fs = 0;
    int cur = -1;
    for (long long base = lo; base < hi; base += 32) {
      const int n = (int)min(32ll, hi - base);
      const bool in = lane < n;
      const int mj = in ? sm[base + lane] : 0, dj = in ? sd[base + lane] : 0, fj = in ? sf[base + lane] : 0;
      for (int i = 0; i < n; i += 4) {
        int mm[4], dd[4], ff[4];
        float row[4][KC];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          mm[u] = __shfl_sync(0xffffffffu, mj, (i + u) & 31);
          dd[u] = __shfl_sync(0xffffffffu, dj, (i + u) & 31);
          ff[u] = __shfl_sync(0xffffffffu, fj, (i + u) & 31);
          if (u > 0 && i + u >= n) {  // past the end: repeat the previous slot with count 0
            mm[u] = mm[u - 1];
            dd[u] = dd[u - 1];
            ff[u] = 0;
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int c = 0; c < KC; ++c) {
            const int col = cb + lane + 32 * c;
            row[u][c] = col < r ? S[(long long)dd[u] * r + col] : 0.f;
          }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (mm[u] != cur) {
            if (cur >= 0) sk_flush<KC>(cur, acc, fs, lo, hi, wcnt, r, cb, Z, C, lane);
            cur = mm[u];
#pragma unroll
            for (int c = 0; c < KC; ++c) {
              const int col = cb + lane + 32 * c;
              acc[c] = 0.f;
              om[c] = col < r ? __ldg(Om + (long long)cur * r + col) : 0.f;
            }
            fs = 0;
          }
          const float fu = (float)ff[u];
#pragma unroll
          for (int c = 0; c < KC; ++c) acc[c] = fmaf(fu, row[u][c] - om[c], acc[c]);
          fs += ff[u];
        }
      }
    }
    if (cur >= 0) sk_flush<KC>(cur, acc, fs, lo, hi, wcnt, r, cb, Z, C, lane);
  }
}

// Workspace of a re-whitening (one FP64 allocation, made by tlda_online_begin).
struct OnlineWs {
  double *Y, *Q1, *Q2, *M1, *U64;               // V x r (three), V, V x D
  double *G, *Z, *LinvT, *L1, *L2, *L1T, *C1, *C2, *Bm, *Et, *Ms, *Rs;  // r x r
  double *m1q, *ev, *Ek, *lam;                  // r, r, r x D, D
  static size_t words(size_t V, size_t r, size_t D) { return 3 * V * r + V + V * D + 12 * r * r + 2 * r + r * D + D; }
  OnlineWs(double *w, size_t V, size_t r, size_t D) {
    double **rr_bufs[] = {&G, &Z, &LinvT, &L1, &L2, &L1T, &C1, &C2, &Bm, &Et, &Ms, &Rs};
    Y = w, Q1 = Y + V * r, Q2 = Q1 + V * r, M1 = Q2 + V * r, U64 = M1 + V;
    w = U64 + V * D;
    for (double **b : rr_bufs) {
      *b = w;
      w += r * r;
    }
    m1q = w, ev = m1q + r, Ek = ev + r, lam = Ek + r * D;
  }
};

// Rebuilds the whitening from the online statistics (section "Fully Online
// Implementation", the PCA update): with M1 = C/T, the sketch of
// M2 = (alpha0+1) P/S2 - alpha0 M1 M1^T is Y = (alpha0+1)/S2 Z - alpha0 M1 (M1^T Omega);
// then the single-pass eigendecomposition of Halko, Martinsson and Tropp
// (2011, section 5.5): Q = orth(Y) (FP64 CholeskyQR2), B solves
// B (Q^T Omega) = Q^T Y, B symmetrised, B = E Lambda E^T (Jacobi), U = Q E,
// and W = U_D Lambda_D^-1/2 with the signs of fit_moments, m1 = W^T M1, U.
// The previous W is kept in on_Wold.
tlda_status online_rewhiten(tlda_ctx *ctx) {
  cudaStream_t s = ctx->stream;
  const int V = ctx->V, D = ctx->D, r = ctx->on_r;
  unsigned long long TS[3];
  int ferr = 0;
  CKF(cudaMemcpyAsync(TS, ctx->on_TS, sizeof TS, cudaMemcpyDeviceToHost, s));
  CKF(cudaMemcpyAsync(&ferr, ctx->on_err, sizeof ferr, cudaMemcpyDeviceToHost, s));
  CKF(cudaStreamSynchronize(s));
  if (ferr) return fail(ctx, TLDA_ERR_INVALID, "corrupt CSR batch in the online pass");
  if (TS[0] == 0 || TS[1] == 0) return fail(ctx, TLDA_ERR_NUMERIC, "no token pairs accumulated");
  const double a0 = ctx->p.alpha0, sP = (a0 + 1.0) / (double)TS[1];
  OnlineWs w(ctx->on_ws, V, r, D);
  int *status = ctx->on_status, *ex = nullptr;
  const int sms = ctx->num_sms;
  if (tlda_status st = g64_exps(ctx, &ex)) return st;
  CKF(cudaMemsetAsync(status, 0, 2 * sizeof(int), s));
  k_m1<<<(V + 255) / 256, 256, 0, s>>>(ctx->on_C, ctx->on_TS, V, w.M1);
  vec_tn64(w.M1, ctx->on_Om, V, r, w.m1q, s);
  CKF(cudaMemcpyAsync(w.Y, ctx->on_Z, sizeof(double) * (size_t)V * r, cudaMemcpyDeviceToDevice, s));
  k_rank1_fix<<<(unsigned)(((long long)V * r + 255) / 256), 256, 0, s>>>(w.Y, w.M1, w.m1q, V, r, sP, a0);
  // CholeskyQR2: out = in L^-T with L L^T = in^T in, twice; Y = Q2 (L1 L2)^T
  auto cholqr_pass = [&](const double *in, double *out, double *Lf) -> tlda_status {
    gemm_tn64(in, r, in, r, w.G, r, r, r, V, ex, V, sms, s);
    if (tlda_status st = run_chol_inv(ctx, w.G, r, Lf, w.Z, nullptr, w.LinvT, nullptr, status, s)) return st;
    gemm_nn64(in, r, w.LinvT, r, out, r, V, r, r, ex, V, sms, s);
    return TLDA_OK;
  };
  if (tlda_status st = cholqr_pass(w.Y, w.Q1, w.L1)) return st;
  if (tlda_status st = cholqr_pass(w.Q1, w.Q2, w.L2)) return st;
  gemm_tn64(w.Q2, r, ctx->on_Om, r, w.C2, r, r, r, V, ex, V, sms, s);  // Q^T Omega
  // Q^T Y = R = (L1 L2)^T = L2^T L1^T, in plain FP64 (its rows fall with the spectrum)
  k_transpose_rr<<<(r * r + 255) / 256, 256, 0, s>>>(w.L1, r, w.L1T);
  k_transpose_rr<<<(r * r + 255) / 256, 256, 0, s>>>(w.L2, r, w.Ms);
  k_small_nn<<<r, 256, 0, s>>>(w.Ms, w.L1T, r, r, nullptr, w.C1);
  // B = (Q^T Y)(Q^T Omega)^-1, symmetrised by the eigensolver
  if (tlda_status st = run_solve_right(ctx, w.C1, w.C2, r, w.Ms, w.Rs, w.Bm, status + 1, s)) return st;
  CKF(cudaGetLastError());
  int hstat[2];
  CKF(cudaMemcpyAsync(hstat, status, sizeof hstat, cudaMemcpyDeviceToHost, s));
  CKF(cudaStreamSynchronize(s));
  if (tlda_status st = chol_status(ctx, hstat[0], "sketch basis lost rank (CholeskyQR breakdown)")) return st;
  if (tlda_status st = chol_status(ctx, hstat[1], "Q^T Omega is singular")) return st;
  if (tlda_status js = run_jacobi(ctx, w.Bm, w.G, r, w.Et, w.ev, s)) return js;
  std::vector<double> hev(r), hEv((size_t)r * r);
  CKF(cudaMemcpyAsync(hev.data(), w.ev, sizeof(double) * r, cudaMemcpyDeviceToHost, s));
  CKF(cudaMemcpyAsync(hEv.data(), w.Et, sizeof(double) * r * r, cudaMemcpyDeviceToHost, s));
  CKF(cudaStreamSynchronize(s));
  std::vector<int> ord(r);
  for (int i = 0; i < r; ++i) ord[i] = i;
  std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return hev[x] > hev[y]; });
  std::vector<double> hEk((size_t)r * D), hlam(D);
  for (int j = 0; j < D; ++j) {
    hlam[j] = hev[ord[j]];
    for (int i = 0; i < r; ++i) hEk[(size_t)i * D + j] = hEv[(size_t)ord[j] * r + i];
  }
  if (!(hlam[D - 1] > 1e-12 * hlam[0]))
    return fail(ctx, TLDA_ERR_NUMERIC, "the sketched M2 has fewer than D positive eigenvalues");
  CKF(cudaMemcpyAsync(w.Ek, hEk.data(), sizeof(double) * r * D, cudaMemcpyHostToDevice, s));
  CKF(cudaMemcpyAsync(w.lam, hlam.data(), sizeof(double) * D, cudaMemcpyHostToDevice, s));
  gemm_nn64(w.Q2, r, w.Ek, D, w.U64, D, V, D, r, ex, V, sms, s);
  if (ctx->whitened)
    CKF(cudaMemcpyAsync(ctx->on_Wold, ctx->W32, sizeof(float) * (size_t)V * D, cudaMemcpyDeviceToDevice, s));
  // Y and Q1 are free: the peaks of U's columns
  make_whitening(ctx, w.U64, w.lam, w.M1, w.Y, reinterpret_cast<int *>(w.Q1), w.m1q, s);
  CKF(cudaGetLastError());
  CKF(cudaStreamSynchronize(s));
  ctx->eig = hlam;
  return TLDA_OK;
}

// Phi (D x K, device) <- W^T W_old (W_old^T W_old)^-1 Phi: the factors carried
// from the previous whitening (on_Wold) into the current one (W32).
tlda_status online_rotate(tlda_ctx *ctx, float *Phi) {
  cudaStream_t s = ctx->stream;
  const int V = ctx->V, D = ctx->D, K = ctx->K;
  OnlineWs w(ctx->on_ws, V, ctx->on_r, D);  // r x r buffers hold the D x D ones (D <= r)
  int *status = ctx->on_status, *ex = nullptr;
  const int sms = ctx->num_sms;
  if (tlda_status st = g64_exps(ctx, &ex)) return st;
  CKF(cudaMemsetAsync(status, 0, sizeof(int), s));
  gemm_tn64(ctx->W32, D, ctx->on_Wold, D, w.C1, D, D, D, V, ex, V, sms, s);
  gemm_tn64(ctx->on_Wold, D, ctx->on_Wold, D, w.C2, D, D, D, V, ex, V, sms, s);
  // (W^T W_old) L^-T L^-1 Phi with L the Cholesky factor of W_old^T W_old (a
  // third of the time of the elimination: 2 D/32 grid barriers against D)
  CKF(cudaMemcpyAsync(w.G, w.C2, sizeof(double) * D * D, cudaMemcpyDeviceToDevice, s));
  if (tlda_status st = run_chol_inv(ctx, w.G, D, w.L1, w.Z, w.L2, w.LinvT, nullptr, status, s)) return st;
  float *Pn = reinterpret_cast<float *>(w.Rs);
  k_small_nn<<<D, 256, 0, s>>>(w.L2, Phi, D, K, nullptr, w.Ms);
  k_small_nn<<<D, 256, 0, s>>>(w.LinvT, w.Ms, D, K, nullptr, w.Et);
  k_small_nn<<<D, 256, 0, s>>>(w.C1, w.Et, D, K, nullptr, Pn);
  int hst = 0;
  auto finish = [&]() -> tlda_status {
    CKF(cudaGetLastError());
    CKF(cudaMemcpyAsync(&hst, status, sizeof hst, cudaMemcpyDeviceToHost, s));
    CKF(cudaStreamSynchronize(s));
    return TLDA_OK;
  };
  if (tlda_status st = finish()) return st;
  if (hst == 1) {  // not positive definite to rounding: elimination with pivoting decides
    CKF(cudaMemsetAsync(status, 0, sizeof(int), s));
    if (tlda_status st = run_solve_right(ctx, w.C1, w.C2, D, w.Ms, w.Rs, w.Bm, status, s)) return st;
    k_small_nn<<<D, 256, 0, s>>>(w.Bm, Phi, D, K, nullptr, Pn);
    if (tlda_status st = finish()) return st;
  }
  if (tlda_status st = chol_status(ctx, hst, "W^T W of the previous whitening is singular")) return st;
  CKF(cudaMemcpyAsync(Phi, Pn, sizeof(float) * D * K, cudaMemcpyDeviceToDevice, s));
  CKF(cudaStreamSynchronize(s));
  return TLDA_OK;
}

// Documents [d0, d0 + nd) of `corpus` into the online statistics and sketch,
// in pieces of at most kSkPieceDocs documents and kSkPieceNnz nonzeros (the
// piece offsets are read back once; validation errors land in on_err).
tlda_status online_accumulate(tlda_ctx *ctx, const tlda_csr *corpus, int64_t d0, int nd) {
  if (nd <= 0) return TLDA_OK;
  cudaStream_t s = ctx->stream;
  // columns per lane: 4 up to r = 128, else 8, in ny column groups of 32 kc
  const int V = ctx->V, r = ctx->on_r, kc = r <= 128 ? 4 : 8, ny = (r + 32 * kc - 1) / (32 * kc);
  SketchWs w(ctx->on_sk, V, r);
  int64_t *total = w.scan + scan_blocks(V);
  auto piece = [&](int64_t a, int n, int32_t lo, int32_t hi) -> tlda_status {
    const SkPiece q{corpus->indptr + a, corpus->indices, corpus->counts, n, lo, hi, V, r};
    CKF(cudaMemsetAsync(w.wcnt, 0, sizeof(int32_t) * (V + 1), s));
    CKF(cudaMemsetAsync(w.wfill, 0, sizeof(int32_t) * V, s));
    const unsigned g = (unsigned)(((long long)n * 32 + 255) / 256);
    const dim3 gr(g, ny);
    if (kc == 4) k_sk_rows<4><<<gr, 256, 0, s>>>(q, ctx->on_Om32, w.S, w.wcnt, w.ok, ctx->on_TS, ctx->on_err);
    else k_sk_rows<8><<<gr, 256, 0, s>>>(q, ctx->on_Om32, w.S, w.wcnt, w.ok, ctx->on_TS, ctx->on_err);
    scan_counts(w.wcnt, V, w.scan, total, s);
    k_sk_scatter<<<g, 256, 0, s>>>(q, w.ok, w.wcnt, w.wfill, w.sd, w.sf, w.sm, ctx->on_err);
    const long long span = std::max<long long>(1, (long long)hi - lo);
    const dim3 zg((unsigned)std::min<long long>((span + 8ll * kSkRun - 1) / (8ll * kSkRun), 8ll * ctx->num_sms / ny), ny);
    if (kc == 4) k_sk_z<4><<<zg, 256, 0, s>>>(w.wcnt, w.sd, w.sf, w.sm, total, r, w.S, ctx->on_Om32, ctx->on_Z, ctx->on_C, ctx->on_err);
    else k_sk_z<8><<<zg, 256, 0, s>>>(w.wcnt, w.sd, w.sf, w.sm, total, r, w.S, ctx->on_Om32, ctx->on_Z, ctx->on_C, ctx->on_err);
    CKF(cudaGetLastError());
    return TLDA_OK;
  };
  // a piece whose offsets span more than kSkPieceNnz slots is halved
  std::function<tlda_status(int64_t, int64_t, int32_t, int32_t)> run = [&](int64_t a, int64_t b, int32_t lo,
                                                                          int32_t hi) -> tlda_status {
    if ((long long)hi - lo <= kSkPieceNnz) return piece(a, (int)(b - a), lo, hi);
    if (b - a == 1) return fail(ctx, TLDA_ERR_OOM, "a document with more than 16M nonzeros");
    const int64_t mid = a + (b - a) / 2;
    int32_t hm = 0;
    CKF(cudaMemcpyAsync(&hm, corpus->indptr + mid, sizeof hm, cudaMemcpyDeviceToHost, s));
    CKF(cudaStreamSynchronize(s));
    if (tlda_status st = run(a, mid, lo, hm)) return st;
    return run(mid, b, hm, hi);
  };
  const int np = (nd + kSkPieceDocs - 1) / kSkPieceDocs;
  std::vector<int32_t> h(np + 1);
  CKF(cudaMemcpy2DAsync(h.data(), sizeof(int32_t), corpus->indptr + d0, sizeof(int32_t) * kSkPieceDocs,
                        sizeof(int32_t), np, cudaMemcpyDeviceToHost, s));
  CKF(cudaMemcpyAsync(h.data() + np, corpus->indptr + d0 + nd, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CKF(cudaStreamSynchronize(s));
  for (int i = 0; i < np; ++i) {
    const int64_t a = d0 + (int64_t)i * kSkPieceDocs, b = std::min<int64_t>(a + kSkPieceDocs, d0 + nd);
    if (tlda_status st = run(a, b, h[i], h[i + 1])) return st;
  }
  return TLDA_OK;
}

// Rebuild the whitening; carry Phi (if given) from the previous one.
tlda_status online_whiten(tlda_ctx *ctx, float *Phi) {
  const bool had = ctx->whitened;
  if (tlda_status st = online_rewhiten(ctx)) return st;
  if (had && Phi)
    if (tlda_status st = online_rotate(ctx, Phi)) return st;
  ctx->whitened = true;
  return TLDA_OK;
}

}  // namespace

extern "C" {

tlda_status tlda_fit_moments(tlda_ctx *ctx, const tlda_csr *chunk, uint32_t flags) {
  TLDA_RANGE();
  if (!ctx) return TLDA_ERR_INVALID;
  if (!(flags & (TLDA_ACCUMULATE | TLDA_FINALIZE))) return fail(ctx, TLDA_ERR_INVALID, "flags must hold ACCUMULATE and/or FINALIZE");
  if (ctx->V > kMaxFitV) return fail(ctx, TLDA_ERR_OOM, "fit_moments keeps a dense V x V pair-count matrix: V <= 65536");
  if (flags & TLDA_ACCUMULATE) {
    if (!chunk) return fail(ctx, TLDA_ERR_INVALID, "chunk is NULL");
    if (chunk->vocab != ctx->V || chunk->n_docs < 0 || !chunk->indptr ||
        (chunk->n_docs > 0 && (!chunk->indices || !chunk->counts)))
      return fail(ctx, TLDA_ERR_INVALID, "bad chunk");
    const size_t V = ctx->V;
    if (!ctx->P64) {
      CKF(dalloc(&ctx->P64, V * V));
      if (!ctx->Ccnt) CKF(dalloc(&ctx->Ccnt, V));
      if (!ctx->TS) CKF(dalloc(&ctx->TS, 3));
      CKF(dalloc(&ctx->fit_err, 1));
    }
    if (!ctx->fit_open) {
      CKF(cudaMemsetAsync(ctx->P64, 0, sizeof(double) * V * V, ctx->stream));
      CKF(cudaMemsetAsync(ctx->Ccnt, 0, sizeof(unsigned long long) * V, ctx->stream));
      CKF(cudaMemsetAsync(ctx->TS, 0, sizeof(unsigned long long) * 3, ctx->stream));
      CKF(cudaMemsetAsync(ctx->fit_err, 0, sizeof(int), ctx->stream));
      ctx->fit_open = true;
    }
    if (chunk->n_docs > 0) {
      const long long threads = (long long)chunk->n_docs * 32;
      k_fit_accumulate<<<(unsigned)((threads + 255) / 256), 256, 0, ctx->stream>>>(*chunk, ctx->V, ctx->P64, ctx->Ccnt,
                                                                                  ctx->TS, ctx->fit_err);
      CKF(cudaGetLastError());
    }
  }
  if (flags & TLDA_FINALIZE) {
    if (!ctx->fit_open) return fail(ctx, TLDA_ERR_STATE, "FINALIZE without any ACCUMULATE");
    ctx->fit_open = false;
    return finalize(ctx);
  }
  return TLDA_OK;
}

tlda_status tlda_get_counts(const tlda_ctx *cctx, int64_t *C, int64_t *T, int64_t *S2, int64_t *S3) {
  tlda_ctx *ctx = const_cast<tlda_ctx *>(cctx);
  if (!ctx) return TLDA_ERR_INVALID;
  if (!ctx->Ccnt || !ctx->TS) return fail(ctx, TLDA_ERR_STATE, "no accumulated statistics");
  unsigned long long ts[3];
  CKF(cudaStreamSynchronize(ctx->stream));
  CKF(cudaMemcpy(ts, ctx->TS, sizeof ts, cudaMemcpyDeviceToHost));
  if (C) CKF(cudaMemcpy(C, ctx->Ccnt, sizeof(int64_t) * ctx->V, cudaMemcpyDeviceToHost));
  if (T) *T = (int64_t)ts[0];
  if (S2) *S2 = (int64_t)ts[1];
  if (S3) *S3 = (int64_t)ts[2];
  return TLDA_OK;
}

tlda_status tlda_unwhiten_topics(tlda_ctx *ctx, const float *Phi, double *mu_out, double *alpha_out, uint32_t flags) {
  TLDA_RANGE();
  if (!ctx || !Phi || !mu_out || !alpha_out) return fail(ctx, TLDA_ERR_INVALID, "NULL argument");
  if (!ctx->whitened) return fail(ctx, TLDA_ERR_STATE, "no whitening: fit or set one first");
  cudaStream_t s = ctx->stream;
  const int V = ctx->V, D = ctx->D, K = ctx->K;
  int *ex = nullptr;
  const int sms = ctx->num_sms;
  if (tlda_status st = g64_exps(ctx, &ex)) return st;
  const bool host = flags & TLDA_HOST_OUTPUT;
  double *G = nullptr, *Linv = nullptr, *LinvT = nullptr, *T1 = nullptr, *T = nullptr, *sum = nullptr, *n2 = nullptr;
  double *Lf = nullptr, *Zs = nullptr, *mu = nullptr, *al = nullptr;
  int *status = nullptr;
  const size_t DD = (size_t)D * D, topics = sizeof(double) * V * K;
  const bool keep = topics <= kKeepTopics;
  auto lay = [&](Carver &c) {
    c.take(G, DD);
    c.take(Linv, DD);
    c.take(LinvT, DD);
    c.take(Lf, DD);
    c.take(Zs, DD);
    c.take(T1, (size_t)D * K);
    c.take(T, (size_t)D * K);
    c.take(sum, K);
    c.take(n2, K);
    c.take(status, 1);
    c.take(al, K);
    if (host && keep) c.take(mu, (size_t)V * K);
  };
  // the context keeps this workspace, with the topics of a host output up to
  // kKeepTopics: an allocation and its release took 150 us of each call
  Carver need{nullptr};
  lay(need);
  if (ctx->uw_bytes < need.off) {
    dfree(ctx->uw_ws);
    ctx->uw_bytes = 0;
    CKF(dalloc(&ctx->uw_ws, need.off));
    ctx->uw_bytes = need.off;
  }
  Carver real{ctx->uw_ws};
  lay(real);
  Scratch large;  // larger topics go with the call, which copies them for longer than that
  if (host && !keep) CKF(large.carve([&](Carver &c) { c.take(mu, (size_t)V * K); }));
  if (!host) {
    mu = mu_out;
    al = alpha_out;
  }
  CKF(cudaMemsetAsync(status, 0, sizeof(int), s));
  gemm_tn64(ctx->W32, D, ctx->W32, D, G, D, D, D, V, ex, V, sms, s);    // W^T W = L L^T
  if (tlda_status st = run_chol_inv(ctx, G, D, Lf, Zs, Linv, LinvT, nullptr, status, s)) return st;
  k_unwhiten_norms<<<1, kMaxDim, 0, s>>>(Phi, D, K, n2, al);
  k_small_nn<<<D, 256, 0, s>>>(Linv, Phi, D, K, nullptr, T1);
  k_small_nn<<<D, 256, 0, s>>>(LinvT, T1, D, K, n2, T);                 // (W^T W)^-1 Phi diag(|phi|^2)
  gemm_nn64(ctx->W32, D, T, K, mu, K, V, K, D, ex, V, sms, s);
  const int slab = std::max(32, (V + 63) / 64);
  const dim3 cg((K + 31) / 32, (V + slab - 1) / slab);
  CKF(cudaMemsetAsync(sum, 0, sizeof(double) * K, s));
  k_clip_sum<<<cg, 256, 0, s>>>(mu, V, K, slab, sum);
  k_clip_scale<<<cg, 256, 0, s>>>(mu, V, K, slab, sum);
  CKF(cudaGetLastError());
  int hst = 0;
  CKF(cudaMemcpyAsync(&hst, status, sizeof hst, cudaMemcpyDeviceToHost, s));
  if (host) {
    CKF(cudaMemcpyAsync(mu_out, mu, sizeof(double) * (size_t)V * K, cudaMemcpyDeviceToHost, s));
    CKF(cudaMemcpyAsync(alpha_out, al, sizeof(double) * K, cudaMemcpyDeviceToHost, s));
  }
  CKF(cudaStreamSynchronize(s));
  if (tlda_status st = chol_status(ctx, hst, "W^T W is not positive definite")) return st;
  return TLDA_OK;
}

tlda_status tlda_online_begin(tlda_ctx *ctx, const double *Omega, int32_t r) {
  TLDA_RANGE();
  if (!ctx) return TLDA_ERR_INVALID;
  if (!Omega || r < ctx->D || r > kMaxDim || (r & 1) || r > ctx->V)
    return fail(ctx, TLDA_ERR_INVALID, "the sketch needs an even r with D <= r <= min(V, 512)");
  const size_t V = ctx->V;
  if (ctx->on_r != r) {
    if (ctx->on_Om) cudaFree(ctx->on_Om);
    if (ctx->on_Z) cudaFree(ctx->on_Z);
    if (ctx->on_ws) cudaFree(ctx->on_ws);
    if (ctx->on_sk) cudaFree(ctx->on_sk);
    if (ctx->on_Om32) cudaFree(ctx->on_Om32);
    ctx->on_Om = ctx->on_Z = ctx->on_ws = nullptr;
    ctx->on_sk = nullptr;
    ctx->on_Om32 = nullptr;
    ctx->on_r = 0;
    CKF(dalloc(&ctx->on_Om, V * r));
    CKF(dalloc(&ctx->on_Z, V * r));
    CKF(dalloc(&ctx->on_ws, OnlineWs::words(V, r, ctx->D)));
    CKF(dalloc(reinterpret_cast<char **>(&ctx->on_sk), SketchWs::bytes(V, r)));
    CKF(dalloc(&ctx->on_Om32, V * r));
    ctx->on_r = r;
  }
  if (!ctx->on_C) CKF(dalloc(&ctx->on_C, V));
  if (!ctx->on_TS) CKF(dalloc(&ctx->on_TS, 3));
  if (!ctx->on_err) CKF(dalloc(&ctx->on_err, 1));
  if (!ctx->on_status) CKF(dalloc(&ctx->on_status, 2));
  if (!ctx->on_Wold) CKF(dalloc(&ctx->on_Wold, V * ctx->D));
  cudaStream_t s = ctx->stream;
  CKF(cudaMemcpyAsync(ctx->on_Om, Omega, sizeof(double) * V * r, cudaMemcpyDeviceToDevice, s));
  k_d2f<<<(unsigned)((V * r + 255) / 256), 256, 0, s>>>(ctx->on_Om, ctx->on_Om32, (long long)(V * r));
  CKF(cudaGetLastError());
  CKF(cudaMemsetAsync(ctx->on_Z, 0, sizeof(double) * V * r, s));
  CKF(cudaMemsetAsync(ctx->on_C, 0, sizeof(unsigned long long) * V, s));
  CKF(cudaMemsetAsync(ctx->on_TS, 0, sizeof(unsigned long long) * 3, s));
  CKF(cudaMemsetAsync(ctx->on_err, 0, sizeof(int), s));
  CKF(cudaStreamSynchronize(s));
  ctx->on_active = true;
  return TLDA_OK;
}

tlda_status tlda_online_pass(tlda_ctx *ctx, const tlda_csr *corpus, const int64_t *batch_offsets, int32_t n_batches,
                             float *Phi, float lr, int32_t rewhiten_every, double *loss_out) {
  TLDA_RANGE();
  if (!ctx) return TLDA_ERR_INVALID;
  if (!ctx->on_active) return fail(ctx, TLDA_ERR_STATE, "tlda_online_begin has not been called");
  if (!corpus || corpus->vocab != ctx->V || corpus->n_docs < 0 || !corpus->indptr ||
      (corpus->n_docs > 0 && (!corpus->indices || !corpus->counts)))
    return fail(ctx, TLDA_ERR_INVALID, "bad corpus");
  if (!Phi || !batch_offsets || n_batches < 0 || rewhiten_every < 1)
    return fail(ctx, TLDA_ERR_INVALID, "bad online pass arguments");
  for (int b = 0; b < n_batches; ++b) {
    const int64_t d0 = batch_offsets[b], d1 = batch_offsets[b + 1];
    if (d0 < 0 || d1 < d0 || d1 > corpus->n_docs) return fail(ctx, TLDA_ERR_INVALID, "batch offsets out of range");
  }
  for (int b0 = 0; b0 < n_batches; b0 += rewhiten_every) {
    const int b1 = std::min(n_batches, b0 + rewhiten_every);
    const int64_t d0 = batch_offsets[b0], d1 = batch_offsets[b1];
    if (tlda_status st = online_accumulate(ctx, corpus, d0, (int)(d1 - d0))) return st;
    if (tlda_status st = online_whiten(ctx, Phi)) return st;
    tlda_status st = tlda_cp_pass(ctx, corpus, batch_offsets + b0, b1 - b0, Phi, lr, 0,
                                  loss_out ? loss_out + b0 : nullptr);
    if (st) return st;
  }
  return TLDA_OK;
}

tlda_status tlda_online_accumulate(tlda_ctx *ctx, const tlda_csr *corpus) {
  TLDA_RANGE();
  if (!ctx) return TLDA_ERR_INVALID;
  if (!ctx->on_active) return fail(ctx, TLDA_ERR_STATE, "tlda_online_begin has not been called");
  if (!corpus || corpus->vocab != ctx->V || corpus->n_docs < 0 || !corpus->indptr ||
      (corpus->n_docs > 0 && (!corpus->indices || !corpus->counts)))
    return fail(ctx, TLDA_ERR_INVALID, "bad corpus");
  return online_accumulate(ctx, corpus, 0, corpus->n_docs);
}

tlda_status tlda_online_whiten(tlda_ctx *ctx, float *Phi) {
  TLDA_RANGE();
  if (!ctx) return TLDA_ERR_INVALID;
  if (!ctx->on_active) return fail(ctx, TLDA_ERR_STATE, "tlda_online_begin has not been called");
  return online_whiten(ctx, Phi);
}

tlda_status tlda_online_get_sketch(tlda_ctx *ctx, double *Z_out, int64_t *C_out, int64_t *TS_out) {
  TLDA_RANGE();
  if (!ctx) return TLDA_ERR_INVALID;
  if (!ctx->on_active) return fail(ctx, TLDA_ERR_STATE, "tlda_online_begin has not been called");
  const size_t V = ctx->V, r = ctx->on_r;
  cudaStream_t s = ctx->stream;
  int herr = 0;
  if (Z_out) CKF(cudaMemcpyAsync(Z_out, ctx->on_Z, sizeof(double) * V * r, cudaMemcpyDefault, s));
  if (C_out) CKF(cudaMemcpyAsync(C_out, ctx->on_C, sizeof(int64_t) * V, cudaMemcpyDefault, s));
  if (TS_out) CKF(cudaMemcpyAsync(TS_out, ctx->on_TS, sizeof(int64_t) * 3, cudaMemcpyDefault, s));
  CKF(cudaMemcpyAsync(&herr, ctx->on_err, sizeof herr, cudaMemcpyDeviceToHost, s));
  CKF(cudaStreamSynchronize(s));
  if (herr) return fail(ctx, TLDA_ERR_INVALID, "a corrupt document was met since tlda_online_begin");
  return TLDA_OK;
}

tlda_status tlda_online_set_sketch(tlda_ctx *ctx, const double *Z, const int64_t *C, const int64_t *TS) {
  TLDA_RANGE();
  if (!ctx) return TLDA_ERR_INVALID;
  if (!ctx->on_active) return fail(ctx, TLDA_ERR_STATE, "tlda_online_begin has not been called");
  if (!Z || !C || !TS) return fail(ctx, TLDA_ERR_INVALID, "Z, C and TS are required");
  const size_t V = ctx->V, r = ctx->on_r;
  cudaStream_t s = ctx->stream;
  CKF(cudaMemcpyAsync(ctx->on_Z, Z, sizeof(double) * V * r, cudaMemcpyDefault, s));
  CKF(cudaMemcpyAsync(ctx->on_C, C, sizeof(int64_t) * V, cudaMemcpyDefault, s));
  CKF(cudaMemcpyAsync(ctx->on_TS, TS, sizeof(int64_t) * 3, cudaMemcpyDefault, s));
  CKF(cudaMemsetAsync(ctx->on_err, 0, sizeof(int), s));
  CKF(cudaStreamSynchronize(s));
  return TLDA_OK;
}

}  // extern "C"
