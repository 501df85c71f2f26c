// Hot-path kernels of the online Tensor LDA CP step (eq. vec_deriv and the SGD
// update of section "Online Learning of the Third Moment"), plain FP32 form,
// plus the pieces both precisions share: the touched words, batch scan +
// whitening, the Phi-only terms and the final reduction/update.
//
// Per step, with U = W - 1 m1^T (V x D), X = F U, Y = X Phi, Q = U Phi:
//   touched words {m : c_m > 0}, c_m = sum_d f_dm          k_touch
//   a7/a8  G3, P = Phi (Phi^T Phi * Phi^T Phi)             k_phi_gram, k_phi_terms
//   a9  grad = E - 3 c3/S3 (G1 + G2), Phi -= lr grad       k_reduce_update
// where E = 3(1+theta) P - 3 G3, and the data term G1 + G2 in one of two ways.
//
// FP32 without the loss: the sums regrouped by word,
//   a4  Q = U Phi (touched rows)                           k_q_f32
//   a1  CSR validation, S3;  y_d = sum_j f_j q_j,  r_d = sum_j f_j q_j^2,
//       z_d = y_d^2 - r_d,  B_m += f_j (z_d + 2 q_j^2 - 2 q_j y_d)   k_doc
//   a5+a6  G1 + G2 = U^T B over the touched words          k_gw_f32
// X, Y, Z and their rows of the two products are not formed: the sum is
// G1 + G2 = sum_j u_j [f_j (z + 2 q_j^2 - 2 q_j y)]^T term by term.
//
// With the loss (its FP32 sums keep their order) and in the BF16 form:
//   a1  L_d, S3, CSR validation;  a2  X = F U (= F W - L m1^T)  k_scan_whiten
//   a3  Y = X Phi;  a4 Q = U Phi (touched rows)            k_qy_f32
//   a4  R_d = sum_m f_dm Q_m^2,  Z = Y*Y - R;  H = F^T Y   k_rz
//   a6  Zc_m = Q_m * (2 c_m Q_m - 2 H_m)                   k_zh_f32
//   a5+a6  G1 + G2 = X^T Z + U^T Zc (split reduction)      k_g_f32
// Words a batch does not touch have c_m = 0 and H_m = 0 (B_m = 0), so they
// contribute nothing to G2 and are skipped.
//
// H (or B) and c take one add per nonzero.  A word that most documents hold
// (the head of a Zipf vocabulary) would queue every document's add at one
// address, so small tables are kept nrep times (StepArgs::nrep): a block adds
// to one copy, and the reader sums them (batches of few documents use one).
#include <algorithm>
#include <cstdio>

#include "tlda_internal.h"

namespace tlda {

__device__ __forceinline__ float4 f4(float x) { return make_float4(x, x, x, x); }
__device__ __forceinline__ float4 fma4(float s, float4 a, float4 c) {
  return make_float4(fmaf(s, a.x, c.x), fmaf(s, a.y, c.y), fmaf(s, a.z, c.z), fmaf(s, a.w, c.w));
}

// ------------------------------------------------------------ batch descriptor
__global__ void k_set_desc(DevState *st, BatchDesc b) { st->cur = b; }

__global__ void k_begin_pass(DevState *st, const BatchDesc *descs, int n) {
  st->descs = descs;
  st->n_descs = n;
  st->pass_pos = 1;
  st->cur = descs[0];
}

void launch_set_desc(DevState *st, const BatchDesc &b, cudaStream_t s) {
  k_set_desc<<<1, 1, 0, s>>>(st, b);
}
void launch_begin_pass(DevState *st, const BatchDesc *descs, int n, cudaStream_t s) {
  k_begin_pass<<<1, 1, 0, s>>>(st, descs, n);
}

// ------------------------------------------------------------ U = W - 1 m1^T
__global__ void k_make_u(const float *W, const float *m1, int V, int D, int Dp, float *U32,
                         __nv_bfloat16 *U16) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)V * Dp) return;
  const int m = (int)(e / Dp), i = (int)(e % Dp);
  const float u = i < D ? W[(long long)m * D + i] - m1[i] : 0.f;
  U32[e] = u;
  if (U16) U16[e] = __float2bfloat16_rn(u);
}

void launch_make_u(const float *W, const float *m1, int V, int D, int Dp, float *U32,
                   __nv_bfloat16 *U16, cudaStream_t s) {
  const long long n = (long long)V * Dp;
  k_make_u<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(W, m1, V, D, Dp, U32, U16);
}

// ------------------------------------------------------------ a1 + a2: scan and whiten
// Nonzeros of one document, 32 at a time: lane j holds nonzero base + j (word,
// count), checked in place; invalid entries get weight 0 on row 0.
struct NzChunk {
  int m, f;      // word (0 if invalid) and count (0 if invalid)
  bool in;       // lane holds a nonzero of this chunk
  bool bad;      // lane's nonzero breaks the CSR rules
  int n;         // nonzeros in this chunk (same in all lanes)
};

__device__ __forceinline__ NzChunk load_chunk(const BatchDesc &b, int V, int base, int hi, int lane, int prev) {
  NzChunk c;
  const int j = base + lane;
  c.in = j < hi;
  c.n = min(32, hi - base);
  int m = -1, f = 0;
  if (c.in) {
    m = __ldg(b.indices + ((long long)j - b.nz_base));
    f = __ldg(b.counts + ((long long)j - b.nz_base));
  }
  int mp = __shfl_up_sync(0xffffffffu, m, 1);
  if (lane == 0) mp = prev;
  const bool valid = c.in && m >= 0 && m < V && f > 0;
  c.bad = c.in && (!valid || m <= mp);
  c.m = valid ? m : 0;
  c.f = valid ? f : 0;
  return c;
}

// Whether document row [lo, hi) lies in the batch's nonzero range (the offsets
// at its first and last document): outside it the row offsets decrease
// somewhere, and k_touch has not seen the words.  Nor has it where the batch's
// first offset is out of range: then no row is taken.
__device__ __forceinline__ bool row_in_batch(const BatchDesc &b, int lo, int hi, int first, int last) {
  return first >= b.nz_base && lo >= first && hi >= lo && hi <= last;
}

// Touched words of the batch into widx (compact, no fixed order) with flag set.
// A word's first meeting in a block goes to its flag, the others end at the
// block's bitmap (a word that most documents hold would else queue thousands of
// exchanges at one address: 11.7 us a batch of 4096 tweets).  Flat over the nonzeros, four
// a thread of the NT and turn; a word already flagged costs one load, not an atomic; one add
// to n_touched a block and turn.
constexpr int kTouchBits = 1 << 17;  // words a block's bitmap holds (16 KB); larger vocabularies do without
template <int NT>
__device__ void touch_words(const StepArgs &a, const BatchDesc &b, int *n_touched, int block, int blocks) {
  if (b.n_docs <= 0) return;
  const int lo = b.indptr[0], hi = b.indptr[b.n_docs];
  if (lo < b.nz_base || hi < lo) return;  // corrupt: k_doc / k_scan_whiten report it
  __shared__ int wsum[NT / 32], base;
  __shared__ unsigned seen[kTouchBits / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool small = a.V <= kTouchBits;
  if ((long long)lo + (long long)block * (4 * NT) >= hi) return;
  if (small) {
    for (int i = tid; i < (a.V + 31) / 32; i += NT) seen[i] = 0;
    __syncthreads();
  }
  for (long long j0 = (long long)lo + (long long)block * (4 * NT); j0 < hi; j0 += (long long)blocks * (4 * NT)) {
    int m[4];
    unsigned fresh = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long j = j0 + u * NT + tid;
      m[u] = j < hi ? __ldg(b.indices + (j - b.nz_base)) : -1;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (m[u] < 0 || m[u] >= a.V) continue;
      if (small) {
        const unsigned bit = 1u << (m[u] & 31);
        if (atomicOr(&seen[m[u] >> 5], bit) & bit) continue;
      }
      if (*reinterpret_cast<volatile int *>(a.flag + m[u]) == 0 && atomicExch(a.flag + m[u], 1) == 0) fresh |= 1u << u;
    }
    const int mine = __popc(fresh);
    int pre = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, pre, o);
      if (lane >= o) pre += y;
    }
    if (lane == 31) wsum[w] = pre;
    __syncthreads();
    if (tid == 0) {
      int t = 0;
#pragma unroll
      for (int q = 0; q < NT / 32; ++q) {
        const int x = wsum[q];
        wsum[q] = t;
        t += x;
      }
      base = t ? atomicAdd(n_touched, t) : 0;
    }
    __syncthreads();
    int at = base + wsum[w] + pre - mine;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (fresh & (1u << u)) a.widx[at++] = m[u];
    __syncthreads();  // wsum, base
  }
}

__global__ void __launch_bounds__(256) k_touch(StepArgs a) {
  touch_words<256>(a, a.st->cur, &a.st->n_touched, blockIdx.x, gridDim.x);
}

// The same for a batch given by value, which becomes the step's batch.
__global__ void __launch_bounds__(256) k_touch_batch(StepArgs a, BatchDesc b) {
  if (blockIdx.x == 0 && threadIdx.x == 0) a.st->cur = b;
  touch_words<256>(a, b, &a.st->n_touched, blockIdx.x, gridDim.x);
}

// Blocks of 256 threads that find the touched words beside other work (one turn each at 32 nonzeros a document).
int touch_blocks(const StepArgs &a) { return std::max(64, std::min(2 * a.sms, a.Bmax / 32)); }

void launch_touch(const StepArgs &a, cudaStream_t s) { k_touch<<<2 * a.sms, 256, 0, s>>>(a); }
void launch_touch_batch(const StepArgs &a, const BatchDesc &b, cudaStream_t s) {
  k_touch_batch<<<std::min(2 * a.sms, b.n_docs / 8 + 1), 256, 0, s>>>(a, b);  // 128 nonzeros a document: one turn
}

// Four U rows q .. q + 3 of a chunk into acc (FP32, in the chunk's order).
template <int NV>
__device__ __forceinline__ void add_rows(const NzChunk &c, int q, const float *U32, int Dp, int cols, int lane,
                                         float4 (&acc)[NV]) {
  int mm[4];
  float ff[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    mm[u] = __shfl_sync(0xffffffffu, c.m, (q + u) & 31);
    ff[u] = (float)__shfl_sync(0xffffffffu, c.f, (q + u) & 31);
    if (q + u >= c.n) ff[u] = 0.f;
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int col = v * 128 + lane * 4;
    if (col < cols) {
      float4 r[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) r[u] = __ldg(reinterpret_cast<const float4 *>(U32 + (long long)mm[u] * Dp + col));
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[v] = fma4(ff[u], r[u], acc[v]);
    }
  }
}

// One warp per document: validates the row, accumulates L_d and
// x_d = sum_m f_dm u_m (FP32) four U rows in flight at a time, adds c_m to this
// block's copy and the block's share of S3.  TC=true writes X in BF16 row-major
// (X16), whole rows, else in FP32.  The first `touch` blocks (FP32 only) find the
// batch's touched words meanwhile: the product after this kernel reads them.  Up
// to 128 features two blocks an SM are asked for: without that the compiler takes
// 40 registers and spills, 2 to 3 us a step.
template <int NV, bool TC>
__global__ void __launch_bounds__(32 * kDocsPerBlock, NV == 1 ? 2 : 0) k_scan_whiten(StepArgs a, int touch) {
  const BatchDesc b = a.st->cur;
  if constexpr (!TC)
    if ((int)blockIdx.x < touch) return touch_words<32 * kDocsPerBlock>(a, b, &a.st->n_touched, blockIdx.x, touch);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, block = blockIdx.x - touch;
  const int d0 = block * kDocsPerBlock;
  if (d0 >= (TC ? round_up(b.n_docs, 64) : b.n_docs)) return;
  const int d = d0 + warp;
  __shared__ unsigned long long s3;
  if (threadIdx.x == 0) s3 = 0;
  __syncthreads();
  const int copy = (block & (copies(a, b.n_docs) - 1)) * a.V;  // this block's counts start there
  float4 acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = f4(0.f);
  if (d < b.n_docs) {
    const int lo = b.indptr[d], hi = b.indptr[d + 1];
    bool bad = !row_in_batch(b, lo, hi, b.indptr[0], b.indptr[b.n_docs]);
    long long lsum = 0;
    int prev = -1;
    if (!bad) {
      for (int base = lo; base < hi; base += 32) {
        const NzChunk c = load_chunk(b, a.V, base, hi, lane, prev);
        if (__any_sync(0xffffffffu, c.bad)) bad = true;
        prev = __shfl_sync(0xffffffffu, c.in ? c.m : -1, c.n - 1);
        lsum += c.f;
        if (a.same_token && c.f > 0) atomicAdd(a.cnt + (copy + c.m), c.f);
        for (int q = 0; q < c.n; q += 4) add_rows<NV>(c, q, a.U32, a.Dp, a.Dp, lane, acc);
      }
    }
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    const long long L = lsum;
    if (bad && lane == 0) atomicOr(&a.st->err, kErrCsr);
    if (lane == 0 && L >= 3) atomicAdd(&s3, (unsigned long long)(L * (L - 1) * (L - 2)));
    if (!TC) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int col = v * 128 + lane * 4;
        if (col < a.Dp) *reinterpret_cast<float4 *>(a.X32 + (long long)d * a.Dp + col) = acc[v];
      }
    }
  }
  if constexpr (TC) {
    if (d < round_up(b.n_docs, 64)) {
      // row-major BF16 copy: the A operand of Y = X Phi and of G1 = X^T Z (rows
      // past the batch, up to the next multiple of 64, are written as zeros)
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int col = v * 128 + lane * 4;
        if (col < a.Dp) {
          __nv_bfloat162 p[2] = {__floats2bfloat162_rn(acc[v].x, acc[v].y), __floats2bfloat162_rn(acc[v].z, acc[v].w)};
          *reinterpret_cast<uint2 *>(a.X16 + (long long)d * a.Dp + col) = *reinterpret_cast<const uint2 *>(p);
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && s3) atomicAdd(&a.st->S3, s3);
}

void launch_whiten(const StepArgs &a, cudaStream_t s) {
  const bool tc = a.precision == TLDA_BF16;
  const int touch = !tc && a.same_token ? touch_blocks(a) * 256 / (32 * kDocsPerBlock) : 0;
  const int grid = touch + round_up(a.Bmax, 64) / kDocsPerBlock;
  const int nv = (a.Dp + 127) / 128;
#define TLDA_WHITEN(NVv)                                                              \
  if (nv == NVv) {                                                                    \
    if (tc) k_scan_whiten<NVv, true><<<grid, 32 * kDocsPerBlock, 0, s>>>(a, touch);   \
    else k_scan_whiten<NVv, false><<<grid, 32 * kDocsPerBlock, 0, s>>>(a, touch);     \
    return;                                                                           \
  }
  TLDA_WHITEN(1) TLDA_WHITEN(2) TLDA_WHITEN(3) TLDA_WHITEN(4)
#undef TLDA_WHITEN
}

// X = F U of one batch given by value into the caller's B x D array
// (tlda_whiten_batch): no step state but the error bits.  One warp per document,
// bound by the latency of its dependent loads (offsets, nonzeros, rows): small
// blocks sized to the batch, only the D columns of a row read, and whole 16-byte
// stores where the output's rows allow them (`wide`).  8192 documents at D = 100:
// 15.0 -> 9.3 us a call; the kernel shared with the CP step needed its batch
// written to the step state by a launch of its own and stored 4 bytes a lane.
template <int NV>
__global__ void __launch_bounds__(128) k_whiten_out(BatchDesc b, int V, int D, int Dp, const float *__restrict__ U32, int *err,
                                                    float *__restrict__ X, int wide) {
  const int d = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (d >= b.n_docs) return;
  const int lo = b.indptr[d], hi = b.indptr[d + 1], cols = (D + 3) & ~3;
  bool bad = lo < b.nz_base || hi < lo;
  float4 acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = f4(0.f);
  if (!bad) {
    int prev = -1;
    for (int base = lo; base < hi; base += 32) {
      const NzChunk c = load_chunk(b, V, base, hi, lane, prev);
      bad |= __any_sync(0xffffffffu, c.bad);
      prev = __shfl_sync(0xffffffffu, c.in ? c.m : -1, c.n - 1);
#pragma unroll 4
      for (int q = 0; q < c.n; q += 4) add_rows<NV>(c, q, U32, Dp, cols, lane, acc);
    }
  }
  if (bad && lane == 0) atomicOr(err, kErrCsr);
  float *x = X + (long long)d * D;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int col = v * 128 + lane * 4;
    if (wide) {
      if (col < D) *reinterpret_cast<float4 *>(x + col) = acc[v];
    } else {
      const float c[4] = {acc[v].x, acc[v].y, acc[v].z, acc[v].w};
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (col + q < D) x[col + q] = c[q];
    }
  }
}

void launch_whiten_out(const StepArgs &a, const BatchDesc &b, cudaStream_t s, float *X) {
  const int grid = (b.n_docs + 3) / 4, nv = (a.Dp + 127) / 128;
  const int wide = a.D % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
  if (nv == 1) k_whiten_out<1><<<grid, 128, 0, s>>>(b, a.V, a.D, a.Dp, a.U32, &a.st->err, X, wide);
  else if (nv == 2) k_whiten_out<2><<<grid, 128, 0, s>>>(b, a.V, a.D, a.Dp, a.U32, &a.st->err, X, wide);
  else if (nv == 3) k_whiten_out<3><<<grid, 128, 0, s>>>(b, a.V, a.D, a.Dp, a.U32, &a.st->err, X, wide);
  else k_whiten_out<4><<<grid, 128, 0, s>>>(b, a.V, a.D, a.Dp, a.U32, &a.st->err, X, wide);
}

// ------------------------------------------------------------ a7/a8: Phi-only terms
// Gram = Phi^T Phi (Kp x Kp, zero padded) in 32 x 32 tiles over 64-row slabs
// of Phi held in shared memory; the extra block row forms a = m1^T Phi.
__global__ void __launch_bounds__(256) k_phi_gram(StepArgs a) {
  const int bx = blockIdx.x, by = blockIdx.y, tid = threadIdx.x;
  if (by == (int)gridDim.y - 1) {
    if (tid < 32) {
      const int j = bx * 32 + tid;
      float s = 0.f;
      if (j < a.K) {
#pragma unroll 8
        for (int r = 0; r < a.D; ++r) s = fmaf(a.m1[r], a.Phi[(long long)r * a.K + j], s);
      }
      if (j < a.Kp) a.avec[j] = s;
    }
    return;
  }
  __shared__ float Pi[64][33], Pj[64][33];
  const int ii = tid >> 3, jj = (tid & 7) * 4;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int r0 = 0; r0 < a.D; r0 += 64) {
#pragma unroll
    for (int e = tid; e < 64 * 32; e += 256) {
      const int r = e >> 5, c = e & 31, gr = r0 + r;
      const int ci = by * 32 + c, cj = bx * 32 + c;
      Pi[r][c] = (gr < a.D && ci < a.K) ? a.Phi[(long long)gr * a.K + ci] : 0.f;
      Pj[r][c] = (gr < a.D && cj < a.K) ? a.Phi[(long long)gr * a.K + cj] : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int r = 0; r < 64; ++r) {
      const float x = Pi[r][ii];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fmaf(x, Pj[r][jj + q], acc[q]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) a.Gram[(by * 32 + ii) * a.Kp + bx * 32 + jj + q] = acc[q];
}

// P = Phi (Gram * Gram) in 32 x 32 tiles (rows r of Phi, columns i), then per
// entry G3 = 2 phi_ri a_i + m1_r |phi_i|^2 - 2 m1_r a_i^2 and
// E = 3(1+theta) P - 3 G3.  Block (0, 0) also forms the Phi-only loss part.
__global__ void __launch_bounds__(256) k_phi_terms(StepArgs a) {
  const int bx = blockIdx.x, by = blockIdx.y, tid = threadIdx.x;
  __shared__ float Pr[32][65], G2[64][33];
  const int rr = tid >> 3, ic = (tid & 7) * 4;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int j0 = 0; j0 < a.K; j0 += 64) {
#pragma unroll
    for (int e = tid; e < 32 * 64; e += 256) {
      const int r = e >> 6, j = e & 63, gr = by * 32 + r, gj = j0 + j;
      Pr[r][j] = (gr < a.D && gj < a.K) ? a.Phi[(long long)gr * a.K + gj] : 0.f;
      const int jb = e >> 5, c = e & 31, gjb = j0 + jb, gi = bx * 32 + c;
      const float g = (gjb < a.K && gi < a.K) ? a.Gram[gjb * a.Kp + gi] : 0.f;
      G2[jb][c] = g * g;
    }
    __syncthreads();
#pragma unroll 8
    for (int j = 0; j < 64; ++j) {
      const float x = Pr[rr][j];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fmaf(x, G2[j][ic + q], acc[q]);
    }
    __syncthreads();
  }
  const int r = by * 32 + rr;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = bx * 32 + ic + q;
    if (r < a.D && i < a.K) {
      const float ai = a.avec[i], n2 = a.Gram[i * a.Kp + i], mr = a.m1[r];
      const float g3 = 2.f * a.Phi[(long long)r * a.K + i] * ai + mr * n2 - 2.f * mr * ai * ai;
      a.G3[r * a.Kp + i] = g3;
      a.E[r * a.Kp + i] = 3.f * (1.f + a.theta) * acc[q] - 3.f * g3;
    }
  }
  if (bx == 0 && by == 0 && a.want_loss) {
    __shared__ double red[256];
    double s = 0.0;
    for (int q = tid; q < a.K * a.K; q += blockDim.x) {
      const double g = a.Gram[(q / a.K) * a.Kp + (q % a.K)];
      s += 0.5 * (1.0 + a.theta) * g * g * g;
    }
    for (int i = tid; i < a.K; i += blockDim.x) {
      const double ai = a.avec[i], n2 = a.Gram[i * a.Kp + i];
      s -= 3.0 * ai * n2 - 2.0 * ai * ai * ai;
    }
    red[tid] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
      if (tid < w) red[tid] += red[tid + w];
      __syncthreads();
    }
    if (tid == 0) a.st->loss_phi = red[0];
  }
}

void launch_phi_gram(const StepArgs &a, cudaStream_t s) {
  dim3 g(a.Kp / 32, a.Kp / 32 + 1);
  k_phi_gram<<<g, 256, 0, s>>>(a);
}

void launch_phi_terms(const StepArgs &a, cudaStream_t s) {
  dim3 g(a.Kp / 32, a.Dp / 32);
  k_phi_terms<<<g, 256, 0, s>>>(a);
}

// ------------------------------------------------------------ Phi^T image (BF16 forms)
__global__ void k_phi_img(StepArgs a) { phi_img_groups(a, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x); }

void launch_phi_img(const StepArgs &a, cudaStream_t s) { k_phi_img<<<16, 256, 0, s>>>(a); }

// ------------------------------------------------------------ a3/a4: Q and Y (FP32)
// Rows t < n_touched: Q[widx[t]] = U[widx[t]] Phi; then Y[d] = X[d] Phi.
// 64 x 64 output tile per block, 4 x 4 per thread, Phi read with bounds
// straight from the caller's D x K layout (zero padding).
__global__ void __launch_bounds__(256) k_qy_f32(StepArgs a) {
  const int nt = a.same_token ? a.st->n_touched : 0;
  const int rows = nt + a.st->cur.n_docs;
  const int r0 = blockIdx.x * 64;
  if (r0 >= rows) return;
  const int n0 = blockIdx.y * 64;
  __shared__ __align__(16) float As[32][68];
  __shared__ __align__(16) float Bs[32][64];
  __shared__ const float *arow[64];
  __shared__ float *orow[64];
  const int tid = threadIdx.x;
  if (tid < 64) {
    const int r = r0 + tid;
    const float *ap = nullptr;
    float *op = nullptr;
    if (r < nt) {
      const int m = a.widx[r];
      ap = a.U32 + (long long)m * a.Dp;
      op = a.Q32 + (long long)m * a.Kp;
    } else if (r < rows) {
      const int d = r - nt;
      ap = a.X32 + (long long)d * a.Dp;
      op = a.Y32 + (long long)d * a.Kp;
    }
    arow[tid] = ap;
    orow[tid] = op;
  }
  __syncthreads();
  const int tx = tid & 15, ty = tid >> 4;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  for (int k0 = 0; k0 < a.Dp; k0 += 32) {
    {
      const int r = tid >> 2, kk = (tid & 3) * 8;
      const float *ap = arow[r];
      float4 v0 = f4(0.f), v1 = f4(0.f);
      if (ap) {
        v0 = *reinterpret_cast<const float4 *>(ap + k0 + kk);
        v1 = *reinterpret_cast<const float4 *>(ap + k0 + kk + 4);
      }
      As[kk + 0][r] = v0.x; As[kk + 1][r] = v0.y; As[kk + 2][r] = v0.z; As[kk + 3][r] = v0.w;
      As[kk + 4][r] = v1.x; As[kk + 5][r] = v1.y; As[kk + 6][r] = v1.z; As[kk + 7][r] = v1.w;
    }
    for (int e = tid; e < 32 * 64; e += 256) {
      const int kk = e >> 6, n = e & 63, gi = k0 + kk, gn = n0 + n;
      Bs[kk][n] = (gi < a.D && gn < a.K) ? a.Phi[(long long)gi * a.K + gn] : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < 32; ++kk) {
      const float4 av = *reinterpret_cast<const float4 *>(&As[kk][ty * 4]);
      const float4 bv = *reinterpret_cast<const float4 *>(&Bs[kk][tx * 4]);
      const float ar[4] = {av.x, av.y, av.z, av.w}, br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float *op = orow[ty * 4 + i];
    if (op) *reinterpret_cast<float4 *>(op + n0 + tx * 4) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  }
}

// ------------------------------------------------------------ a4 + a6 scatter: R, Z, H
// One warp per document (8 per block: small blocks keep more warps resident
// per SM): r_d = sum_m f_dm q_m^2 over gathered Q rows (four in flight),
// z_d = y_d^2 - r_d, H_m += f_dm y_d (vector atomics), and the document part
// of the loss.  TC=true writes Z as whole BF16 rows (Z16), zero rows past the
// batch up to the next multiple of 64.
template <int NK, bool TC>
__global__ void __launch_bounds__(256) k_rz(StepArgs a) {
  const BatchDesc b = a.st->cur;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int d0 = blockIdx.x * 8, d = d0 + warp;
  if (d0 >= (TC ? round_up(b.n_docs, 64) : b.n_docs)) return;
  const int K4 = (a.K + 3) & ~3;  // Q, Y and H are zero in the padding columns
  float4 y[NK], r[NK];
#pragma unroll
  for (int v = 0; v < NK; ++v) {
    const int col = v * 128 + lane * 4;
    y[v] = (d < b.n_docs && col < a.Kp) ? *reinterpret_cast<const float4 *>(a.Y32 + (long long)d * a.Kp + col)
                                         : f4(0.f);
    r[v] = f4(0.f);
  }
  float *H = a.H32 + (long long)(blockIdx.x & (copies(a, b.n_docs) - 1)) * a.V * a.Kp;
  if (a.same_token && d < b.n_docs) {
    const int lo = b.indptr[d], hi = b.indptr[d + 1];
    if (row_in_batch(b, lo, hi, b.indptr[0], b.indptr[b.n_docs])) {
      for (int base = lo; base < hi; base += 32) {
        const NzChunk c = load_chunk(b, a.V, base, hi, lane, -1);
        for (int q = 0; q < c.n; q += 4) {
          int mm[4];
          float ff[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            mm[u] = __shfl_sync(0xffffffffu, c.m, (q + u) & 31);
            ff[u] = (float)__shfl_sync(0xffffffffu, c.f, (q + u) & 31);
            if (q + u >= c.n) ff[u] = 0.f;
          }
          // all NK x 4 row pieces are requested before the first H atomic (loads
          // are not moved across the atomics by the compiler)
          float4 qv[NK][4];
#pragma unroll
          for (int v = 0; v < NK; ++v) {
            const int col = v * 128 + lane * 4;
#pragma unroll
            for (int u = 0; u < 4; ++u)
              qv[v][u] = col < K4 ? *reinterpret_cast<const float4 *>(a.Q32 + (long long)mm[u] * a.Kp + col)
                                    : f4(0.f);
          }
#pragma unroll
          for (int v = 0; v < NK; ++v) {
            const int col = v * 128 + lane * 4;
            if (col < K4) {
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const float ff2 = ff[u];
                r[v].x = fmaf(ff2 * qv[v][u].x, qv[v][u].x, r[v].x);
                r[v].y = fmaf(ff2 * qv[v][u].y, qv[v][u].y, r[v].y);
                r[v].z = fmaf(ff2 * qv[v][u].z, qv[v][u].z, r[v].z);
                r[v].w = fmaf(ff2 * qv[v][u].w, qv[v][u].w, r[v].w);
                if (ff2 != 0.f)
                  atomicAdd(reinterpret_cast<float4 *>(H + (long long)mm[u] * a.Kp + col),
                            make_float4(ff2 * y[v].x, ff2 * y[v].y, ff2 * y[v].z, ff2 * y[v].w));
              }
            }
          }
        }
      }
    }
  }
  float ls = 0.f;
#pragma unroll
  for (int v = 0; v < NK; ++v) {
    const int col = v * 128 + lane * 4;
    if (col < a.Kp) {
      const float4 z = make_float4(y[v].x * y[v].x - r[v].x, y[v].y * y[v].y - r[v].y,
                                   y[v].z * y[v].z - r[v].z, y[v].w * y[v].w - r[v].w);
      if constexpr (TC) {
        if (d < round_up(b.n_docs, 64)) {
          __nv_bfloat162 p[2] = {__floats2bfloat162_rn(z.x, z.y), __floats2bfloat162_rn(z.z, z.w)};
          *reinterpret_cast<uint2 *>(a.Z16 + (long long)d * a.Kp + col) = *reinterpret_cast<const uint2 *>(p);
        }
      } else {
        if (d < b.n_docs) *reinterpret_cast<float4 *>(a.Z32 + (long long)d * a.Kp + col) = z;
      }
      if (a.want_loss)
        ls += y[v].x * (y[v].x * y[v].x - 3.f * r[v].x) + y[v].y * (y[v].y * y[v].y - 3.f * r[v].y) +
              y[v].z * (y[v].z * y[v].z - 3.f * r[v].z) + y[v].w * (y[v].w * y[v].w - 3.f * r[v].w);
    }
  }
  if (a.want_loss) {
    for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, o);
    if (lane == 0 && ls != 0.f) atomicAdd(&a.st->loss_data, (double)ls);
  }
}

// c_m and four columns of H_m (or B_m), summed over the nrep copies in use.
__device__ __forceinline__ int word_count(const StepArgs &a, int nrep, int m) {
  int c = a.cnt[m];
  for (int r = 1; r < nrep; ++r) c += a.cnt[(long long)r * a.V + m];
  return c;
}
__device__ __forceinline__ float4 word_sum(const StepArgs &a, int nrep, int m, int col) {
  const float4 *p = reinterpret_cast<const float4 *>(a.H32 + (long long)m * a.Kp + col);
  float4 h = *p;
  for (int r = 1; r < nrep; ++r) {
    const float4 x = p[(long long)r * a.V * (a.Kp / 4)];
    h = make_float4(h.x + x.x, h.y + x.y, h.z + x.z, h.w + x.w);
  }
  return h;
}

// ------------------------------------------------------------ a6: Zc rows
// One warp per touched word (compact slot t): Zc_t = q * (2 c q - 2 H_m); then
// H_m, c_m and the flag are cleared for the next batch (this warp is their only
// reader).
template <int NK>
__global__ void __launch_bounds__(256) k_zh_f32(StepArgs a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * 8 + warp;
  if (t >= a.st->n_touched) return;
  const int m = a.widx[t], nrep = copies(a, a.st->cur.n_docs);
  const float c = (float)word_count(a, nrep, m);
  float ls = 0.f;
#pragma unroll
  for (int v = 0; v < NK; ++v) {
    const int col = v * 128 + lane * 4;
    if (col < a.Kp) {
      float4 *hp = reinterpret_cast<float4 *>(a.H32 + (long long)m * a.Kp + col);
      const float4 q = *reinterpret_cast<const float4 *>(a.Q32 + (long long)m * a.Kp + col);
      const float4 h = word_sum(a, nrep, m, col);
      const float4 z = make_float4(q.x * (2.f * c * q.x - 2.f * h.x), q.y * (2.f * c * q.y - 2.f * h.y),
                                   q.z * (2.f * c * q.z - 2.f * h.z), q.w * (2.f * c * q.w - 2.f * h.w));
      *reinterpret_cast<float4 *>(a.Zc32 + (long long)t * a.Kp + col) = z;
      for (int r = 0; r < nrep; ++r) hp[(long long)r * a.V * (a.Kp / 4)] = f4(0.f);
      ls += q.x * q.x * q.x + q.y * q.y * q.y + q.z * q.z * q.z + q.w * q.w * q.w;
    }
  }
  if (a.want_loss) {
    for (int o = 16; o > 0; o >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, o);
    if (lane == 0) atomicAdd(&a.st->loss_data, 2.0 * (double)c * (double)ls);
  }
  __syncwarp();
  if (lane == 0) {
    for (int r = 0; r < nrep; ++r) a.cnt[(long long)r * a.V + m] = 0;
    a.flag[m] = 0;
  }
}

// ------------------------------------------------------------ a5 + a6: G1 + G2 (FP32)
// Split reduction over the rows [docs: (X, Z)] ++ [touched words: (U, Zc)]:
// block (s, ti, tn) sums rows of split s into the 64 x 64 tile (ti, tn) of
// partial s, 4 x 4 outputs per thread.
__global__ void __launch_bounds__(256) k_g_f32(StepArgs a) {
  const int nd = a.st->cur.n_docs, nt = a.same_token ? a.st->n_touched : 0;
  const int R = nd + nt;
  const int s = blockIdx.x, i0 = blockIdx.y * 64, n0 = blockIdx.z * 64;
  const int rb = (int)((long long)R * s / a.nsplit), re = (int)((long long)R * (s + 1) / a.nsplit);
  __shared__ __align__(16) float As[32][64];
  __shared__ __align__(16) float Bs[32][64];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  for (int r0 = rb; r0 < re; r0 += 32) {
    {
      const int rr = tid >> 3, cc = (tid & 7) * 8, r = r0 + rr;
      float4 a0 = f4(0.f), a1 = f4(0.f), b0 = f4(0.f), b1 = f4(0.f);
      if (r < re) {
        const float *ap, *bp;
        if (r < nd) {
          ap = a.X32 + (long long)r * a.Dp;
          bp = a.Z32 + (long long)r * a.Kp;
        } else {
          const int t = r - nd;
          ap = a.U32 + (long long)a.widx[t] * a.Dp;
          bp = a.Zc32 + (long long)t * a.Kp;
        }
        a0 = *reinterpret_cast<const float4 *>(ap + i0 + cc);
        a1 = *reinterpret_cast<const float4 *>(ap + i0 + cc + 4);
        b0 = *reinterpret_cast<const float4 *>(bp + n0 + cc);
        b1 = *reinterpret_cast<const float4 *>(bp + n0 + cc + 4);
      }
      *reinterpret_cast<float4 *>(&As[rr][cc]) = a0;
      *reinterpret_cast<float4 *>(&As[rr][cc + 4]) = a1;
      *reinterpret_cast<float4 *>(&Bs[rr][cc]) = b0;
      *reinterpret_cast<float4 *>(&Bs[rr][cc + 4]) = b1;
    }
    __syncthreads();
#pragma unroll 8
    for (int rr = 0; rr < 32; ++rr) {
      const float4 av = *reinterpret_cast<const float4 *>(&As[rr][ty * 4]);
      const float4 bv = *reinterpret_cast<const float4 *>(&Bs[rr][tx * 4]);
      const float ar[4] = {av.x, av.y, av.z, av.w}, br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
    }
    __syncthreads();
  }
  float *gp = a.Gpart + (long long)s * a.Dp * a.Kp;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<float4 *>(gp + (long long)(i0 + ty * 4 + i) * a.Kp + n0 + tx * 4) =
        make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
}

void launch_qy_f32(const StepArgs &a, cudaStream_t s) {
  dim3 g((a.V + a.Bmax + 63) / 64, a.Kp / 64);
  k_qy_f32<<<g, 256, 0, s>>>(a);
}

void launch_rz(const StepArgs &a, cudaStream_t s) {
  const int nk = (a.Kp + 127) / 128;
  const bool tc = a.precision == TLDA_BF16;
#define TLDA_RZ(NKv)                                                                      \
  if (nk == NKv) {                                                                        \
    if (tc) k_rz<NKv, true><<<round_up(a.Bmax, 64) / 8, 256, 0, s>>>(a);                 \
    else k_rz<NKv, false><<<round_up(a.Bmax, 64) / 8, 256, 0, s>>>(a);                   \
    return;                                                                               \
  }
  TLDA_RZ(1) TLDA_RZ(2) TLDA_RZ(3) TLDA_RZ(4)
#undef TLDA_RZ
}

void launch_zh_f32(const StepArgs &a, cudaStream_t s) {
  const int nk = (a.Kp + 127) / 128;
  if (nk == 1) k_zh_f32<1><<<(a.V + 7) / 8, 256, 0, s>>>(a);
  else if (nk == 2) k_zh_f32<2><<<(a.V + 7) / 8, 256, 0, s>>>(a);
  else if (nk == 3) k_zh_f32<3><<<(a.V + 7) / 8, 256, 0, s>>>(a);
  else k_zh_f32<4><<<(a.V + 7) / 8, 256, 0, s>>>(a);
}

void launch_g_f32(const StepArgs &a, cudaStream_t s) {
  dim3 g(a.nsplit, a.Dp / 64, a.Kp / 64);
  k_g_f32<<<g, 256, 0, s>>>(a);
}

// ------------------------------------------------------------ FP32, by word
// cp.async of one element (4 bytes) or four (16 bytes); zeros where !in.
__device__ __forceinline__ void cp4(float *dst, const float *src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src), "r"(in ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp16(float *dst, const float *src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
               "l"(src), "r"(in ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Two FP32 multiply-adds in one instruction (each rounded as fmaf's): half the
// issue slots of the products below.
__device__ __forceinline__ uint64_t pair(float x, float y) {
  uint64_t p;
  asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(x), "f"(y));
  return p;
}
__device__ __forceinline__ void fma2(uint64_t &c, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpair(uint64_t p) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}

// Q of the touched words: Q[widx[t]] = U[widx[t]] Phi.  Tiles of 64 touched rows
// x 16 TN topics (4 x TN outputs a thread), blocks striding over the tiles.  The
// tile's rows and its part of Phi come to shared memory whole, up to kQDeep
// features at a time, so that a tile waits for memory once and not once a slab;
// a block keeps its part of Phi while its tiles share it.
constexpr int kQDeep = 128, kQRows = 64, kQThreads = 4 * kQRows;
template <int TN>
__global__ void __launch_bounds__(kQThreads) k_q_f32(StepArgs a) {
  constexpr int BN = 16 * TN, LDA = kQDeep + 4;
  extern __shared__ __align__(16) float q_sm[];
  float *As = q_sm, *Bs = q_sm + kQRows * LDA;  // rows x LDA; deep x BN
  const int nt = a.st->n_touched, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int rt = (nt + kQRows - 1) / kQRows, ntn = (a.Kp + BN - 1) / BN, tiles = rt * ntn;
  const bool wide = (a.K & 3) == 0 && (reinterpret_cast<uintptr_t>(a.Phi) & 15) == 0;
  int kept = -1;  // the column tile whose Phi is in Bs (D <= kQDeep)
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int r0 = tile % rt * kQRows, nn = tile / rt, n0 = nn * BN;
    uint64_t acc[4][TN / 2];  // pairs of topics
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0;
    for (int d0 = 0; d0 < a.D; d0 += kQDeep) {
      const int deep = min(kQDeep, (a.D - d0 + 3) & ~3);  // U is zero from D to Dp
      __syncthreads();  // the slab before has been read
      for (int e = tid; e < kQRows * (deep / 4); e += kQThreads) {
        const int r = e / (deep / 4), k = e % (deep / 4) * 4;
        const bool in = r0 + r < nt;
        cp16(As + r * LDA + k, in ? a.U32 + (long long)a.widx[r0 + r] * a.Dp + d0 + k : a.U32, in);
      }
      if (kept != nn || a.D > kQDeep) {
        if (wide) {
          for (int e = tid; e < deep * (BN / 4); e += kQThreads) {
            const int k = e / (BN / 4), n = e % (BN / 4) * 4;
            const bool in = d0 + k < a.D && n0 + n < a.K;
            cp16(Bs + k * BN + n, in ? a.Phi + (long long)(d0 + k) * a.K + n0 + n : a.Phi, in);
          }
        } else {
          for (int e = tid; e < deep * BN; e += kQThreads) {
            const int k = e / BN, n = e % BN;
            const bool in = d0 + k < a.D && n0 + n < a.K;
            cp4(Bs + k * BN + n, in ? a.Phi + (long long)(d0 + k) * a.K + n0 + n : a.Phi, in);
          }
        }
        kept = nn;
      }
      cp_commit();
      cp_wait<0>();
      __syncthreads();
#pragma unroll 2
      for (int k = 0; k < deep; k += 4) {
        float x[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 v = *reinterpret_cast<const float4 *>(As + (ty * 4 + i) * LDA + k);
          x[i][0] = v.x, x[i][1] = v.y, x[i][2] = v.z, x[i][3] = v.w;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint64_t br[TN / 2];
#pragma unroll
          for (int j = 0; j < TN; j += 4) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(Bs + (k + q) * BN + (j / 4) * 64 + tx * 4);
            br[j / 2] = v.x, br[j / 2 + 1] = v.y;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint64_t xx = pair(x[i][q], x[i][q]);
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], xx, br[j]);
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + ty * 4 + i;
      if (r >= nt) continue;
      float *op = a.Q32 + (long long)a.widx[r] * a.Kp;
#pragma unroll
      for (int j = 0; j < TN; j += 4) {
        const int n = n0 + (j / 4) * 64 + tx * 4;
        const float2 lo = unpair(acc[i][j / 2]), hi = unpair(acc[i][j / 2 + 1]);
        if (n < a.Kp) *reinterpret_cast<float4 *>(op + n) = make_float4(lo.x, lo.y, hi.x, hi.y);
      }
    }
  }
}

void launch_q_f32(const StepArgs &a, cudaStream_t s) {
  const int deep = std::min(kQDeep, (a.D + 3) & ~3), rt = (a.V + kQRows - 1) / kQRows;
#define TLDA_Q(TNv, blocks)                                                                               \
  {                                                                                                       \
    const int smem = (kQRows * (kQDeep + 4) + deep * 16 * TNv) * (int)sizeof(float);                          \
    static SmemLimit lim;                                                                                 \
    lim.raise((const void *)k_q_f32<TNv>, (kQRows * (kQDeep + 4) + kQDeep * 16 * TNv) * 4);               \
    k_q_f32<TNv><<<std::min(blocks * a.sms, rt * ((a.Kp + 16 * TNv - 1) / (16 * TNv))), kQThreads, smem, s>>>(a); \
  }
  if (a.Kp % 128 == 64) TLDA_Q(4, 3)
  else TLDA_Q(8, 2)
#undef TLDA_Q
}

// One warp per document, striding: the row's validation, S3, then over its Q rows
// y = sum f q and r = sum f q^2 (z = y^2 - r; r = 0 without the same-token
// correction), and B_m += f (z + 2 q^2 - 2 q y) (f z without it) by vector adds
// into this block's copy.  The rows come by cp.async into the warp's shared
// memory, R of them at once: all of a short document's rows are in flight
// together and are read twice there; a longer one gathers its rows again.
// LW lanes hold a row (8 or 16 up to 32 or 64 topics, else the warp): a narrow
// model's warp takes 32 / LW rows at a time and adds the parts at the end.
template <int NK, int LW>
__global__ void __launch_bounds__(256, NK == 1 ? 4 : 3) k_doc(StepArgs a, int R) {
  constexpr int SUB = 32 / LW, UN = SUB < 4 ? 4 / SUB : 1;  // rows at a time, turns unrolled
  extern __shared__ __align__(16) float doc_rows[];
  const BatchDesc b = a.st->cur;
  if (b.n_docs <= 0) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane / LW, sl = lane % LW;
  const int K4 = (a.K + 3) & ~3;  // the padding columns are zero and stay so
  float *rows = doc_rows + (long long)warp * R * K4;
  float *B = a.H32 + (long long)(blockIdx.x & (copies(a, b.n_docs) - 1)) * a.V * a.Kp;
  const int first = b.indptr[0], last = b.indptr[b.n_docs];
  __shared__ unsigned long long s3;
  if (threadIdx.x == 0) s3 = 0;
  __syncthreads();
  for (int d = blockIdx.x * 8 + warp; d < b.n_docs; d += gridDim.x * 8) {
    const int lo = b.indptr[d], hi = b.indptr[d + 1];
    if (!row_in_batch(b, lo, hi, first, last)) {
      if (lane == 0) atomicOr(&a.st->err, kErrCsr);
      continue;
    }
    bool bad = false;
    long long L = 0;
    float4 y[NK], r[NK];
#pragma unroll
    for (int v = 0; v < NK; ++v) y[v] = r[v] = f4(0.f);
    // rows [s0, s0 + n) of a chunk of nonzeros into shared memory
    auto stage = [&](const NzChunk &c, int s0, int n) {
      for (int j0 = 0; j0 < n; j0 += UN * SUB)
#pragma unroll
        for (int u = 0; u < UN; ++u) {
          const int jj = j0 + u * SUB + sub, j = min(jj, n - 1);
          const float *src = a.Q32 + (long long)__shfl_sync(0xffffffffu, c.m, s0 + j) * a.Kp + sl * 4;
          const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(rows + j * K4 + sl * 4));
#pragma unroll
          for (int v = 0; v < NK; ++v)
            if (jj < n && v * 128 + sl * 4 < K4)
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + v * 512), "l"(src + v * 128) : "memory");
        }
      asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
      __syncwarp();
    };
    const bool once = hi - lo <= min(R, 32);
    NzChunk c{};
    int prev = -1;
    for (int base = lo; base < hi; base += 32) {
      c = load_chunk(b, a.V, base, hi, lane, prev);
      bad |= __any_sync(0xffffffffu, c.bad);
      prev = __shfl_sync(0xffffffffu, c.in ? c.m : -1, c.n - 1);
      L += c.f;
      for (int s0 = 0; s0 < c.n; s0 += R) {
        const int n = min(R, c.n - s0);
        __syncwarp();  // the rows before have been read
        stage(c, s0, n);
        for (int j0 = 0; j0 < n; j0 += UN * SUB)
#pragma unroll
          for (int u = 0; u < UN; ++u) {  // past the end: the last row with count 0
            const int jj = j0 + u * SUB + sub, j = min(jj, n - 1);
            const float fj = (float)__shfl_sync(0xffffffffu, c.f, s0 + j), f = jj < n ? fj : 0.f;
#pragma unroll
            for (int v = 0; v < NK; ++v) {
              const int col = v * 128 + sl * 4;
              if (col < K4) {
                const float4 q = *reinterpret_cast<const float4 *>(rows + j * K4 + col);
                y[v] = fma4(f, q, y[v]);
                r[v].x = fmaf(f * q.x, q.x, r[v].x);
                r[v].y = fmaf(f * q.y, q.y, r[v].y);
                r[v].z = fmaf(f * q.z, q.z, r[v].z);
                r[v].w = fmaf(f * q.w, q.w, r[v].w);
              }
            }
          }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
    if (lane == 0) {
      if (bad) atomicOr(&a.st->err, kErrCsr);
      if (L >= 3) atomicAdd(&s3, (unsigned long long)(L * (L - 1) * (L - 2)));
    }
#pragma unroll
    for (int o = LW; o < 32; o <<= 1) {  // the parts of a narrow model's rows
      const float4 py = y[0], pr = r[0];
      y[0] = make_float4(py.x + __shfl_xor_sync(0xffffffffu, py.x, o), py.y + __shfl_xor_sync(0xffffffffu, py.y, o),
                         py.z + __shfl_xor_sync(0xffffffffu, py.z, o), py.w + __shfl_xor_sync(0xffffffffu, py.w, o));
      r[0] = make_float4(pr.x + __shfl_xor_sync(0xffffffffu, pr.x, o), pr.y + __shfl_xor_sync(0xffffffffu, pr.y, o),
                         pr.z + __shfl_xor_sync(0xffffffffu, pr.z, o), pr.w + __shfl_xor_sync(0xffffffffu, pr.w, o));
    }
    const float on = a.same_token ? 1.f : 0.f;
    float4 z[NK];
#pragma unroll
    for (int v = 0; v < NK; ++v)
      z[v] = make_float4(fmaf(y[v].x, y[v].x, -on * r[v].x), fmaf(y[v].y, y[v].y, -on * r[v].y),
                         fmaf(y[v].z, y[v].z, -on * r[v].z), fmaf(y[v].w, y[v].w, -on * r[v].w));
    const float two = 2.f * on;
    for (int base = lo; base < hi; base += 32) {
      if (!once) c = load_chunk(b, a.V, base, hi, lane, -1);
      for (int s0 = 0; s0 < c.n; s0 += R) {
        const int n = min(R, c.n - s0);
        if (!once) {
          __syncwarp();
          stage(c, s0, n);
        }
        for (int j0 = 0; j0 < n; j0 += UN * SUB)
#pragma unroll
          for (int u = 0; u < UN; ++u) {
            const int jj = j0 + u * SUB + sub, j = min(jj, n - 1);
            const int m = __shfl_sync(0xffffffffu, c.m, s0 + j);
            const float f = (float)__shfl_sync(0xffffffffu, c.f, s0 + j);
            if (jj >= n || f == 0.f) continue;
#pragma unroll
            for (int v = 0; v < NK; ++v) {
              const int col = v * 128 + sl * 4;
              if (col < K4) {
                const float4 q = *reinterpret_cast<const float4 *>(rows + j * K4 + col);
                atomicAdd(reinterpret_cast<float4 *>(B + (long long)m * a.Kp + col),
                          make_float4(f * fmaf(two * q.x, q.x - y[v].x, z[v].x), f * fmaf(two * q.y, q.y - y[v].y, z[v].y),
                                      f * fmaf(two * q.z, q.z - y[v].z, z[v].z), f * fmaf(two * q.w, q.w - y[v].w, z[v].w)));
              }
            }
          }
      }
    }
    __syncwarp();  // the next document's rows
  }
  __syncthreads();
  if (threadIdx.x == 0 && s3) atomicAdd(&a.st->S3, s3);
}

// Rows staged at once: 6.9 KB a warp (17 at K = 100, 32 up to 53 topics), so that
// four blocks of 8 warps fit an SM.
constexpr int kDocBytes = 6912;
void launch_doc(const StepArgs &a, cudaStream_t s) {
  const int K4 = (a.K + 3) & ~3, nk = (a.Kp + 127) / 128;
  const int R = std::max(3, std::min(32, kDocBytes / (K4 * 4)));
  const int smem = 8 * R * K4 * (int)sizeof(float);
  const int grid = std::max(1, std::min((a.Bmax + 7) / 8, 4 * a.sms));
#define TLDA_DOC(NKv, LWv)                                                                                     \
  {                                                                                                            \
    static SmemLimit lim;                                                                                      \
    lim.raise((const void *)k_doc<NKv, LWv>, 8 * kDocBytes);                                                   \
    k_doc<NKv, LWv><<<grid, 256, smem, s>>>(a, R);                                                             \
  }
  if (K4 <= 32) TLDA_DOC(1, 8)
  else if (K4 <= 64) TLDA_DOC(1, 16)
  else if (nk == 1) TLDA_DOC(1, 32)
  else if (nk == 2) TLDA_DOC(2, 32)
  else if (nk == 3) TLDA_DOC(3, 32)
  else TLDA_DOC(4, 32)
#undef TLDA_DOC
}

// Rows t of B summed over the copies into the compact Zc32 (D or K above 128:
// several blocks of k_gw_f32 read a row; a single copy is read where it is);
// k_b_clear clears them afterwards.
__global__ void __launch_bounds__(256) k_b_fold(StepArgs a) {
  const int lane = threadIdx.x & 31;
  for (int t = blockIdx.x * 8 + (threadIdx.x >> 5); t < a.st->n_touched; t += gridDim.x * 8) {
    const int m = a.widx[t];
    for (int col = lane * 4; col < a.Kp; col += 128)
      *reinterpret_cast<float4 *>(a.Zc32 + (long long)t * a.Kp + col) = word_sum(a, copies(a, a.st->cur.n_docs), m, col);
  }
}

// Their rows of B and flags cleared for the next batch (c is not part of this
// form, and need not exist).  A kernel of its own: a warp that loads a row and
// then stores to it waits for the load.
__global__ void __launch_bounds__(256) k_b_clear(StepArgs a) {
  const int lane = threadIdx.x & 31;
  for (int t = blockIdx.x * 8 + (threadIdx.x >> 5); t < a.st->n_touched; t += gridDim.x * 8) {
    const int m = a.widx[t];
    for (int r = 0; r < copies(a, a.st->cur.n_docs); ++r)
      for (int col = lane * 4; col < a.Kp; col += 128)
        *reinterpret_cast<float4 *>(a.H32 + ((long long)r * a.V + m) * a.Kp + col) = f4(0.f);
    if (lane == 0) a.flag[m] = 0;
  }
}

// G1 + G2 = U^T B as a split reduction over the touched rows: block (s, ti, tn)
// sums the rows of split s into a tile of BI features x BN topics of partial s,
// TM x 4 outputs a thread (a warp shares its features; 16 warps at 128 x 128).  Slabs of 16 rows pass through a ring of
// `stages` in shared memory by cp.async: a split has some 90 rows at the usual
// batch sizes, and most of them are requested at once (a slab's arithmetic is
// shorter than a round trip to L2).  FOLD: one tile covers D and K (both at most
// 128), so each row of B has one reader: it sums the copies itself, and clears
// them and the flag for the next batch.
constexpr int kGwRows = 16;
template <int BI, int BN, int TM, bool FOLD>
__global__ void __launch_bounds__(BI / TM * (BN / 4)) k_gw_f32(StepArgs a, int stages) {
  constexpr int TN = 4, TX = BN / TN, NT = BI / TM * TX, BR = kGwRows;
  extern __shared__ __align__(16) float gw_sm[];
  const int reps = FOLD ? copies(a, a.st->cur.n_docs) : 1, stage = BR * (BI + reps * BN);  // at most the host's
  const int nt = a.st->n_touched, tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int s = blockIdx.x, i0 = blockIdx.y * BI, n0 = blockIdx.z * BN;
  const int rb = (int)((long long)nt * s / a.nsplit), re = (int)((long long)nt * (s + 1) / a.nsplit);
  const int slabs = (re - rb + BR - 1) / BR;
  uint64_t acc[TM / 2][TN];  // pairs of features
#pragma unroll
  for (int i = 0; i < TM / 2; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0;
  auto request = [&](int q) {  // slab q into its stage (a group is committed in any case)
    if (q < slabs) {
      float *A = gw_sm + (q % stages) * stage, *B = A + BR * BI;
      const int r0 = rb + q * BR;
#pragma unroll
      for (int i = 0; i < BR * BI / 4 / NT; ++i) {
        const int e = tid + i * NT, r = r0 + e / (BI / 4), c = e % (BI / 4) * 4;
        const bool in = r < re && i0 + c < a.Dp;
        cp16(A + e * 4, in ? a.U32 + (long long)a.widx[r] * a.Dp + i0 + c : a.U32, in);
      }
      for (int p = 0; p < reps; ++p)
#pragma unroll
        for (int i = 0; i < BR * BN / 4 / NT; ++i) {
          const int e = tid + i * NT, r = r0 + e / (BN / 4), c = e % (BN / 4) * 4;
          const bool in = r < re && n0 + c < a.Kp;
          const float *src = a.Zc32;
          if (in)
            src = FOLD || a.nrep == 1 ? a.H32 + ((long long)p * a.V + a.widx[r]) * a.Kp + n0 + c
                                      : a.Zc32 + (long long)r * a.Kp + n0 + c;
          cp16(B + p * BR * BN + e * 4, src, in);
        }
    }
    cp_commit();
  };
  for (int q = 0; q < stages - 1; ++q) request(q);
  for (int q = 0; q < slabs; ++q) {
    // all but the newest stages - 2 groups are there: slab q among them
    switch (stages) {
      case 6: cp_wait<4>(); break;
      case 5: cp_wait<3>(); break;
      case 4: cp_wait<2>(); break;
      case 3: cp_wait<1>(); break;
      default: cp_wait<0>(); break;
    }
    __syncthreads();
    request(q + stages - 1);  // into the stage of slab q - 1, which has been read
    float *A = gw_sm + (q % stages) * stage, *B = A + BR * BI;
    if (FOLD) {
      const int r0 = rb + q * BR;
#pragma unroll
      for (int i = 0; i < BR * BN / 4 / NT; ++i) {
        const int e = tid + i * NT, r = r0 + e / (BN / 4), c = e % (BN / 4) * 4;
        if (reps > 1) {
          float4 v = *reinterpret_cast<float4 *>(B + e * 4);
          for (int p = 1; p < reps; ++p) {
            const float4 x = *reinterpret_cast<const float4 *>(B + p * BR * BN + e * 4);
            v = make_float4(v.x + x.x, v.y + x.y, v.z + x.z, v.w + x.w);
          }
          *reinterpret_cast<float4 *>(B + e * 4) = v;
        }
        if (r < re && c < a.Kp) {
          const int m = a.widx[r];
          for (int p = 0; p < reps; ++p)
            *reinterpret_cast<float4 *>(a.H32 + ((long long)p * a.V + m) * a.Kp + c) = f4(0.f);
          if (c == 0) a.flag[m] = 0;
        }
      }
      if (reps > 1) __syncthreads();
    }
#pragma unroll
    for (int rr = 0; rr < BR; ++rr) {
      uint64_t x[TM / 2];
#pragma unroll
      for (int i = 0; i < TM; i += 4) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(A + rr * BI + (i / 4) * (BI / TM * 4) + ty * 4);
        x[i / 2] = v.x, x[i / 2 + 1] = v.y;
      }
      const float4 v = *reinterpret_cast<const float4 *>(B + rr * BN + tx * 4);
      const uint64_t w[4] = {pair(v.x, v.x), pair(v.y, v.y), pair(v.z, v.z), pair(v.w, v.w)};
#pragma unroll
      for (int i = 0; i < TM / 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) fma2(acc[i][j], x[i], w[j]);
    }
  }
  cp_wait<0>();
  float *gp = a.Gpart + (long long)s * a.Dp * a.Kp;
#pragma unroll
  for (int i = 0; i < TM; i += 2) {
    const int row = i0 + (i / 4) * (BI / TM * 4) + ty * 4 + (i & 3), n = n0 + tx * 4;
    const float2 u[4] = {unpair(acc[i / 2][0]), unpair(acc[i / 2][1]), unpair(acc[i / 2][2]), unpair(acc[i / 2][3])};
    if (row < a.D && n < a.K)
      *reinterpret_cast<float4 *>(gp + (long long)row * a.Kp + n) = make_float4(u[0].x, u[1].x, u[2].x, u[3].x);
    if (row + 1 < a.D && n < a.K)
      *reinterpret_cast<float4 *>(gp + (long long)(row + 1) * a.Kp + n) = make_float4(u[0].y, u[1].y, u[2].y, u[3].y);
  }
}

// Partial sums: one block an SM over the tiles, at least 8; two an SM for the 64 x
// 64 tile, whose block waits more than it computes and whose partial is small, and
// for the 128 x 64 tiles of wide models.
int gw_splits(int Dp, int Kp, int sms) {
  if (Dp > 128 && Kp % 128 == 64) return std::max(8, 2 * sms / ((Dp + 127) / 128 * (Kp / 64)));
  const int tiles = ((Dp + 127) / 128) * ((Kp + 127) / 128);
  return Dp <= 64 ? 2 * sms : std::max(8, sms / tiles);
}

template <int BI, int BN, int TM, bool FOLD>
void gw_launch(const StepArgs &a, dim3 grid, cudaStream_t s) {
  const int stage = kGwRows * (BI + (FOLD ? a.nrep : 1) * BN) * (int)sizeof(float);
  const int stages = std::max(2, std::min(6, 98304 / stage));
  static SmemLimit lim;
  lim.raise((const void *)k_gw_f32<BI, BN, TM, FOLD>, 147456);
  k_gw_f32<BI, BN, TM, FOLD><<<grid, BI / TM * (BN / 4), stages * stage, s>>>(a, stages);
}

void launch_gw_f32(const StepArgs &a, cudaStream_t s) {
  if (a.Dp <= 64) {
    gw_launch<64, 64, 4, true>(a, dim3(a.nsplit), s);
  } else if (a.Dp <= 128 && a.Kp <= 64) {
    gw_launch<128, 64, 8, true>(a, dim3(a.nsplit), s);
  } else if (a.Dp <= 128) {
    gw_launch<128, 128, 8, true>(a, dim3(a.nsplit), s);
  } else {
    if (a.nrep > 1) k_b_fold<<<4 * a.sms, 256, 0, s>>>(a);
    // 64 topics a tile where 128 would compute half a tile of padding (192, 320, 448),
    // as in k_q_f32: V = 65,845, K = 179, us a pass of 8 batches of 5000 documents
    // 2588 -> 2159, of 2000 1521 -> 1284
    if (a.Kp % 128 == 64) gw_launch<128, 64, 8, false>(a, dim3(a.nsplit, (a.Dp + 127) / 128, a.Kp / 64), s);
    else gw_launch<128, 128, 8, false>(a, dim3(a.nsplit, (a.Dp + 127) / 128, (a.Kp + 127) / 128), s);
    k_b_clear<<<4 * a.sms, 256, 0, s>>>(a);
  }
}

// ------------------------------------------------------------ a9: reduce + update
// 32 entries (i, n) per block, the partial sums split over 8 warps:
// g = sum over partials; grad = E - 3 c3/S3 g; Phi -= lr grad (skipped on a
// sticky error or S3 = 0); the BF16 Phi^T image follows Phi.
// Blocks past the entries (a.touch_next of them) take the next batch of a pass
// meanwhile and find its touched words: the flags are clear by now, and nothing
// of that depends on Phi.
__global__ void __launch_bounds__(256) k_reduce_update(StepArgs a) {
  DevState *st = a.st;
  const int entry_blocks = (a.D * a.K + 31) / 32;
  if ((int)blockIdx.x >= entry_blocks && st->descs && st->pass_pos < st->n_descs)
    touch_words<256>(a, st->descs[st->pass_pos], &st->n_touched_next, blockIdx.x - entry_blocks, a.touch_next);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  const unsigned long long S3 = st->S3;
  const int err = st->err;
  // what the end of the step needs besides, requested now by the thread that may do it
  const bool ends = threadIdx.x == 32;
  const BatchDesc *descs = nullptr;
  int pos = 0, n_descs = 0, step = 0;
  double loss_phi = 0.0, loss_data = 0.0;
  if (ends) {
    descs = st->descs, pos = st->pass_pos, n_descs = st->n_descs, step = st->step;
    loss_phi = st->loss_phi, loss_data = st->loss_data;
  }
  const bool live = (int)blockIdx.x < entry_blocks && e < a.D * a.K;
  const int i = live ? e / a.K : 0, n = live ? e % a.K : 0;
  const long long off = (long long)i * a.Kp + n, stride = (long long)a.Dp * a.Kp;
  float part = 0.f;
  if (live) {  // eight partials in flight per iteration
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    int s = w;
    for (; s + 56 < a.nsplit; s += 64) {
#pragma unroll
      for (int u = 0; u < 8; ++u) acc[u] += a.Gpart[(s + 8 * u) * stride + off];
    }
    for (; s < a.nsplit; s += 8) acc[0] += a.Gpart[s * stride + off];
#pragma unroll
    for (int u = 0; u < 8; ++u) part += acc[u];
  }
  const double scale = S3 ? a.c3 / (double)S3 : 0.0;
  const bool more = descs && pos < n_descs;
  BatchDesc next{};
  if (more) next = descs[pos];
  __shared__ float red[8][32];
  red[w][lane] = part;
  __syncthreads();
  if (w == 0 && live) {
    float g = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) g += red[q][lane];
    if (a.mode == 1) {
      a.gdata_out[e] = S3 ? (float)(scale * (double)g) + a.G3[off] : 0.f;
    } else {
      const float grad = S3 ? a.E[off] - (float)(3.0 * scale * (double)g) : 0.f;
      if (a.grad_out) a.grad_out[e] = grad;
      float phi = a.Phi[e];
      if (!err && S3) {
        phi -= a.lr * grad;
        a.Phi[e] = phi;
      }
      if (a.PhiImg) a.PhiImg[phi_img_index(n, i, a.Kp)] = __float2bfloat16_rn(phi);
    }
  }
  // the last block to get here (every block has read the step's sums) ends the
  // step, beside its update: its loss, the sums cleared for the next batch, the step
  // counter, and the next batch descriptor of a pass
  if (ends) {
    unsigned before;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(&st->done) : "memory");
    if (before == gridDim.x - 1) {
      st->n_touched = a.touch_next ? __ldcg(&st->n_touched_next) : 0;
      if (a.touch_next) st->n_touched_next = 0;
      st->done = 0;
      st->loss = S3 ? loss_phi - scale * loss_data : 0.0;
      st->last_S3 = S3;
      st->S3 = 0;
      st->loss_data = 0.0;
      st->step = step + 1;
      if (more) {
        st->cur = next;
        st->pass_pos = pos + 1;
      }
    }
  }
}

void launch_reduce_update(const StepArgs &a, cudaStream_t s) {
  k_reduce_update<<<(a.D * a.K + 31) / 32 + a.touch_next, 256, 0, s>>>(a);
}

}  // namespace tlda
