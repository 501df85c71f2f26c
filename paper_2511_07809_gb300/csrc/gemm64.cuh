// FP64 matrix products on the BF16 tensor cores, by splitting each operand
// into exact whole-number slices (the scheme of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication", Numer. Algorithms 59,
// 2012).
//
//   C = A^T B (tall operands, the Gram matrices) and C = A B (tall times small)
//
// Every row m of op(A) and column n of op(B) gets a power of two 2^e above its
// largest magnitude.  An entry becomes the whole number q = rint(x 2^(55-e)),
// |q| <= 2^55, and q seven balanced base-256 digits d_0 .. d_6 in [-128, 128],
// each exact in BF16.  A product of digits is at most 2^14 in magnitude; the
// digit products of equal order s = i + j are added in one FP32 accumulator,
// at most 7 of them over 128 terms, below 2^24: every sum is exact, whatever
// the order in which the tensor core adds.  After each 128 terms the eight
// accumulators of an entry are folded into two 64-bit integers (order 7 rounded
// to order 6's unit), and at the end into one FP64 value.  Orders s > 7 are
// dropped: per term they are at most 2^-61 of 2^(eA+eB).  Order 7 counts: in
// W^T W of a Zipf vocabulary, whose columns have few large entries, its sum was
// 5e-15 of the result (plain FP64 4e-16, with it 2e-16; 28 digit products a term
// without it, 34 with it).
//
// C = A B sums over columns of A that may differ in scale by many powers of two
// with rows of B the other way round (a whitening and its pseudo-inverse: an
// entry that is small in its row of A then makes a large term).  There term k is
// first scaled, A's column by 2^-c_k and B's row by 2^c_k, with 2^c_k above the
// column's largest magnitude, so that the slices are relative to the terms.
//
// What bounds it, and why: GB300 issues 2 FP64 FMAs a clock per SM (1.2
// TFLOP/s), where the tensor cores take the 34 digit products of a term far
// faster.  Tiles of 64 x 64 by 8 warps (16 x 32 each: 128 accumulators and 32
// 64-bit sums a thread); the raw operands come by cp.async one 32-term slab
// ahead of the products, and are cut into digits in shared memory.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "smem_limit.h"

namespace {

constexpr int kG64Tile = 64;     // rows and columns of C per block
constexpr int kG64Slab = 32;     // terms per shared-memory slab
constexpr int kG64Fold = 128;    // terms per exact FP32 sum
constexpr int kG64Dig = 7;
constexpr int kG64Ord = 8;       // orders of digit products that are summed
constexpr int kG64Ld = kG64Slab + 8;                       // digit row, in BF16 (80 bytes: conflict-free ldmatrix)
constexpr int kG64DigBytes = kG64Dig * kG64Tile * kG64Ld * 2;  // one operand's digits of a slab
constexpr int kG64RawLd = kG64Tile + 1;                    // raw slab row (terms x tile), in elements
constexpr int kG64RawElems = 64 * 33 > kG64Slab * kG64RawLd ? 64 * 33 : kG64Slab * kG64RawLd;
constexpr int kExpNan = 1 << 20;                           // exponent that marks an infinity or NaN
constexpr int kExpZero = -(1 << 16);                       // below that of every number

template <class TA, class TB>
constexpr int g64_smem() {
  return 2 * kG64DigBytes + 2 * kG64RawElems * (int)(sizeof(TA) + sizeof(TB));
}

// Exponent e with |x| < 2^e (FP64 bits); kExpNan for an infinity or NaN,
// kExpZero for zero.
__device__ __forceinline__ int exp_above(double x) {
  const long long b = __double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7ff);
  return E == 0x7ff ? kExpNan : b << 1 == 0 ? kExpZero : E - 1022;  // integer units: an FP64 test takes 64 cycles
}

// e[c] = the largest exp_above over the rows of column c of a rows x cols matrix
// (row pitch ld), each row r first scaled by 2^add[r] when add is given.  FIN:
// infinities and NaN are passed over.  One block per 32 columns and slab of
// rows; e must start below every exponent.
template <bool FIN, class T>
__global__ void __launch_bounds__(256) k_col_exp(const T *x, int ld, int rows, int cols, int slab, const int *add, int *e) {
  __shared__ int red[8][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  const int r0 = blockIdx.y * slab, r1 = min(rows, r0 + slab);
  int m = kExpZero;
  if (c < cols) {
#pragma unroll 8
    for (int r = r0 + w; r < r1; r += 8) {
      const int v = exp_above((double)x[(long long)r * ld + c]);
      if (v == kExpZero) continue;  // add[r] of a term without entries is kExpZero too
      if (v != kExpNan) m = max(m, v + (add ? add[r] : 0));
      else if (!FIN) m = kExpNan;
    }
  }
  red[w][lane] = m;
  __syncthreads();
  if (w == 0 && c < cols) {
#pragma unroll
    for (int q = 1; q < 8; ++q) m = max(m, red[q][lane]);
    atomicMax(e + c, m);
  }
}

// e[r] = the largest exp_above over row r, column c first scaled by 2^-sub[c]:
// one warp per row.
template <class T>
__global__ void __launch_bounds__(256) k_row_exp(const T *x, int ld, int rows, int cols, const int *sub, int *e) {
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (r >= rows) return;
  int m = kExpZero;
#pragma unroll 4
  for (int c = lane; c < cols; c += 32) {
    const int v = exp_above((double)x[(long long)r * ld + c]);
    // a zero has no say in its row's exponent (in a column of zeros v - sub is 0)
    if (v != kExpZero) m = max(m, v == kExpNan ? v : v - sub[c]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) e[r] = m;
}

__device__ __forceinline__ void g64_cp(double *dst, const double *src, bool in) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(in ? 8 : 0) : "memory");
}
__device__ __forceinline__ void g64_cp(float *dst, const float *src, bool in) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(in ? 4 : 0) : "memory");
}

// One operand's raw slab, terms k0 .. k0+31 of tile rows t0 .. t0+63 (past
// kend or nt: zeros, nothing read).  KROWS: the operand is stored with one
// term per row (x[k ld + t]), else one tile row per row (x[t ld + k]).
template <bool KROWS, class T>
__device__ __forceinline__ void g64_load(T *raw, const T *x, int ld, int t0, int nt, int k0, int kend) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int e = threadIdx.x + i * 256;
    const int k = KROWS ? e >> 6 : e & 31, t = KROWS ? e & 63 : e >> 5;
    const bool in = k0 + k < kend && t0 + t < nt;
    const long long at = KROWS ? (long long)(k0 + k) * ld + t0 + t : (long long)(t0 + t) * ld + k0 + k;
    g64_cp(raw + (KROWS ? k * kG64RawLd + t : t * 33 + k), x + (in ? at : 0), in);
  }
}

// The whole number rint(x 2^(55-e)) (half away from zero) plus the bias that
// makes its bytes the balanced digits plus 128 (|x| < 2^e); lo and hi words.
__device__ __forceinline__ uint2 g64_fixed(double x, int e) {
  const int hx = __double2hiint(x);
  const int E = (hx >> 20) & 0x7ff;
  const uint32_t mh = ((uint32_t)hx & 0xfffffu) | (E ? 0x100000u : 0u);
  const unsigned long long m = ((unsigned long long)mh << 32) | (uint32_t)__double2loint(x);
  const int k = max(E, 1) - 1020 - e;  // <= 2 (an infinity or NaN: the result is NaN whatever the digits)
  const unsigned long long q = k > 0 ? m << min(k, 2) : (((m << 1) >> min(-k, 62)) + 1) >> 1;
  const uint32_t neg = (uint32_t)(hx >> 31);
  const unsigned long long s = (q ^ (((unsigned long long)neg << 32) | neg)) + (neg & 1u) + 0x0080808080808080ull;
  return make_uint2((uint32_t)s, (uint32_t)(s >> 32));
}

// Digit of byte i (0: the top) of a pair of fixed values (terms k, k+1) as two
// BF16.  A byte u as FP32 2^23 + u, minus 2^23 + 128: the upper half of that FP32
// is the digit in BF16.  The top digit takes two bytes: it may be 128, 256 with
// the bias.
template <int I>
__device__ __forceinline__ uint32_t g64_digit2(uint2 a, uint2 b) {
  constexpr int byte = 6 - I;
  constexpr uint32_t sel = I == 0 ? 0x7432 : 0x7440 | (byte & 3);  // {0x4b, 0, the upper byte or 0, byte}
  const uint32_t ua = __byte_perm(byte < 4 ? a.x : a.y, 0x4b000000u, sel);
  const uint32_t ub = __byte_perm(byte < 4 ? b.x : b.y, 0x4b000000u, sel);
  const float fa = __uint_as_float(ua) - 8388736.f, fb = __uint_as_float(ub) - 8388736.f;
  return __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
}

// Digits of a raw slab into dig[digit][tile row][term]; SGN * ck[term] is added
// to the exponent of a tile row.
template <bool KROWS, int SGN, class T>
__device__ __forceinline__ void g64_cut(const T *raw, const int *e, const int *ck, __nv_bfloat16 *dig) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int p = threadIdx.x + i * 256, k = (p & 15) * 2, t = p >> 4;
    const int et = e[t];
    const double x0 = (double)raw[KROWS ? k * kG64RawLd + t : t * 33 + k];
    const double x1 = (double)raw[KROWS ? (k + 1) * kG64RawLd + t : t * 33 + k + 1];
    const uint2 a = g64_fixed(x0, SGN ? et + SGN * ck[k] : et), b = g64_fixed(x1, SGN ? et + SGN * ck[k + 1] : et);
    uint32_t *d = reinterpret_cast<uint32_t *>(dig + t * kG64Ld + k);
    constexpr int plane = kG64Tile * kG64Ld / 2;
    d[0] = g64_digit2<0>(a, b);
    d[plane] = g64_digit2<1>(a, b);
    d[2 * plane] = g64_digit2<2>(a, b);
    d[3 * plane] = g64_digit2<3>(a, b);
    d[4 * plane] = g64_digit2<4>(a, b);
    d[5 * plane] = g64_digit2<5>(a, b);
    d[6 * plane] = g64_digit2<6>(a, b);
  }
}

__device__ __forceinline__ void g64_ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

__device__ __forceinline__ void g64_mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// C (M x N, row pitch ldc) = op(A) op(B) over Kd terms; B is stored one term
// per row, A too when AKROWS (C = A^T B), else row-major (C = A B, terms scaled by ck).  eA, eB:
// exponents of the M rows and N columns.  blockIdx.z: split of the terms (in
// whole multiples of kG64Fold); ADD: splits are added into C (zeroed before).
// SYM: A and B are the same, only tiles on or below the diagonal run and each
// is written to both places.
template <bool AKROWS, bool ADD, bool SYM, class TA, class TB>
__global__ void __launch_bounds__(256, 1) k_gemm64(const TA *A, int lda, const TB *B, int ldb, double *C, int ldc,
                                                   int M, int N, int Kd, int chunk, const int *eA, const int *eB, const int *ck) {
  extern __shared__ __align__(16) unsigned char g64_sm[];
  __shared__ int ea[kG64Tile], eb[kG64Tile], cks[2][kG64Slab];
  const int m0 = blockIdx.y * kG64Tile, n0 = blockIdx.x * kG64Tile;
  if (SYM && n0 > m0) return;
  __nv_bfloat16 *dA = reinterpret_cast<__nv_bfloat16 *>(g64_sm), *dB = dA + kG64DigBytes / 2;
  TA *rawA = reinterpret_cast<TA *>(g64_sm + 2 * kG64DigBytes);
  TB *rawB = reinterpret_cast<TB *>(rawA + 2 * kG64RawElems);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, wm = (w & 3) * 16, wn = (w >> 2) * 32;
  const int kb = blockIdx.z * chunk, ke = min(Kd, kb + chunk);
  if (tid < 64) ea[tid] = m0 + tid < M ? eA[m0 + tid] : 0;
  else if (tid < 128) eb[tid - 64] = n0 + tid - 64 < N ? eB[n0 + tid - 64] : 0;
  const bool live = m0 + wm < M && n0 + wn < N;
  float acc[kG64Ord][4][4];
  long long hi[4][4], lo[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      hi[j][q] = lo[j][q] = 0;
#pragma unroll
      for (int s = 0; s < kG64Ord; ++s) acc[s][j][q] = 0.f;
    }
  g64_load<AKROWS>(rawA, A, lda, m0, M, kb, ke);
  g64_load<true>(rawB, B, ldb, n0, N, kb, ke);
  asm volatile("cp.async.commit_group;" ::: "memory");
  const uint32_t sA = static_cast<uint32_t>(__cvta_generic_to_shared(dA)),
                 sB = static_cast<uint32_t>(__cvta_generic_to_shared(dB));
  // ldmatrix rows of this lane: A 16 x 16 (rows 0-15 at terms 0, then at terms
  // 8); B two 8-column groups x 16 terms
  const uint32_t aoff = (uint32_t)(((wm + (lane & 15)) * kG64Ld + (lane >> 4) * 8) * 2);
  const uint32_t boff = (uint32_t)(((wn + (lane & 7) + ((lane >> 4) << 3)) * kG64Ld + ((lane >> 3) & 1) * 8) * 2);
  if (!AKROWS && tid < kG64Slab) cks[0][tid] = kb + tid < ke ? ck[kb + tid] : 0;
  int buf = 0;
  for (int k0 = kb; k0 < ke; k0 += kG64Slab, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // this slab is there; the last slab's digits have been read
    g64_cut<AKROWS, AKROWS ? 0 : 1>(rawA + buf * kG64RawElems, ea, cks[buf], dA);
    g64_cut<true, AKROWS ? 0 : -1>(rawB + buf * kG64RawElems, eb, cks[buf], dB);
    if (k0 + kG64Slab < ke) {
      if (!AKROWS && tid < kG64Slab) {
        const int k = k0 + kG64Slab + tid;
        cks[buf ^ 1][tid] = k < ke ? ck[k] : 0;
      }
      g64_load<AKROWS>(rawA + (buf ^ 1) * kG64RawElems, A, lda, m0, M, k0 + kG64Slab, ke);
      g64_load<true>(rawB + (buf ^ 1) * kG64RawElems, B, ldb, n0, N, k0 + kG64Slab, ke);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    __syncthreads();
    if (!live) continue;
#pragma unroll
    for (int kk = 0; kk < kG64Slab; kk += 16) {
#pragma unroll
      for (int j = 0; j < kG64Dig; ++j) {
        uint32_t b0[4], b1[4];
        const uint32_t bj = sB + boff + (uint32_t)(j * kG64Tile * kG64Ld + kk) * 2;
        g64_ldsm4(b0, bj);
        g64_ldsm4(b1, bj + 16 * kG64Ld * 2);
#pragma unroll
        for (int i = 0; i < kG64Dig && i + j < kG64Ord; ++i) {
          uint32_t a[4];
          g64_ldsm4(a, sA + aoff + (uint32_t)(i * kG64Tile * kG64Ld + kk) * 2);
          g64_mma(acc[i + j][0], a, b0[0], b0[1]);
          g64_mma(acc[i + j][1], a, b0[2], b0[3]);
          g64_mma(acc[i + j][2], a, b1[0], b1[1]);
          g64_mma(acc[i + j][3], a, b1[2], b1[3]);
        }
      }
    }
    if (((k0 - kb) & (kG64Fold - 1)) == kG64Fold - kG64Slab || k0 + kG64Slab >= ke) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          hi[j][q] += ((long long)__float2int_rn(acc[0][j][q]) << 16) + ((long long)__float2int_rn(acc[1][j][q]) << 8) +
                      __float2int_rn(acc[2][j][q]);
          lo[j][q] += ((long long)__float2int_rn(acc[3][j][q]) << 24) + ((long long)__float2int_rn(acc[4][j][q]) << 16) +
                      ((long long)__float2int_rn(acc[5][j][q]) << 8) + __float2int_rn(acc[6][j][q]) +
                      ((__float2int_rn(acc[7][j][q]) + 128) >> 8);
#pragma unroll
          for (int s = 0; s < kG64Ord; ++s) acc[s][j][q] = 0.f;
        }
    }
  }
  __syncthreads();  // ea, eb (an empty range of terms gets here without another barrier)
  if (!live) return;
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int tm = wm + (lane >> 2) + (q >> 1) * 8, tn = wn + j * 8 + (lane & 3) * 2 + (q & 1);
      const int gm = m0 + tm, gn = n0 + tn;
      if (gm >= M || gn >= N || (SYM && gn > gm)) continue;
      // an all-zero row or column has the lowest exponent and sums that are 0
      const int e = ea[tm] + eb[tn];
      double v = scalbn((double)hi[j][q] + (double)lo[j][q] * 0x1p-32, max(e - 30, -4000));
      if (ea[tm] == kExpNan || eb[tn] == kExpNan) v = __longlong_as_double(0x7ff8000000000000ll);
      if (ADD) {
        if (v != 0.0) {
          atomicAdd(C + (long long)gm * ldc + gn, v);
          if (SYM && gn != gm) atomicAdd(C + (long long)gn * ldc + gm, v);
        }
      } else {
        C[(long long)gm * ldc + gn] = v;
      }
    }
}

template <bool AKROWS, bool ADD, bool SYM, class TA, class TB>
void g64_launch(const TA *A, int lda, const TB *B, int ldb, double *C, int ldc, int M, int N, int Kd, int splits,
                const int *eA, const int *eB, const int *ck, cudaStream_t s) {
  static tlda::SmemLimit lim;
  lim.raise((const void *)k_gemm64<AKROWS, ADD, SYM, TA, TB>, g64_smem<TA, TB>());
  const int folds = (Kd + kG64Fold - 1) / kG64Fold, per = (folds + splits - 1) / splits;
  const dim3 g((N + kG64Tile - 1) / kG64Tile, (M + kG64Tile - 1) / kG64Tile, (folds + per - 1) / per);
  k_gemm64<AKROWS, ADD, SYM, TA, TB><<<g, 256, g64_smem<TA, TB>(), s>>>(A, lda, B, ldb, C, ldc, M, N, Kd, per * kG64Fold, eA, eB, ck);
}

}  // namespace
