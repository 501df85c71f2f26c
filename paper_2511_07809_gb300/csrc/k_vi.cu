// Document-topic proportions by variational inference with the topics fixed
// (section "Input and Output": the recovered topic-word matrix and weights
// feed a standard VI; the per-document E-step of Blei, Ng and Jordan 2003,
// section 5.2).  One warp per document, the document's K topics spread over
// the lanes (K/32 each), FP32 throughout.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "tlda.h"
#include "tlda_internal.h"

namespace {

constexpr int kViThreads = 64;  // small blocks: a block's registers are the unit of residence

// digamma(x) for x > 0: below 6 the recurrence psi(x) = psi(x + 6) -
// sum_{i<6} 1/(x + i), the six reciprocals summed as one fraction (pairs
// (a, b) -> (a + b, a b)) and divided once; then the asymptotic series
// ln x - 1/(2x) - sum B_2n / (2n x^2n) (Abramowitz and Stegun 6.3.18)
// through the x^-8 term, whose next term is below 2e-10 at x = 6.
__device__ __forceinline__ float digamma_f(float x) {
  float r = 0.f;
  if (x < 6.f) {
    const float a0 = x, a1 = x + 1.f, a2 = x + 2.f, a3 = x + 3.f, a4 = x + 4.f, a5 = x + 5.f;
    const float n01 = a0 + a1, d01 = a0 * a1, n23 = a2 + a3, d23 = a2 * a3, n45 = a4 + a5, d45 = a4 * a5;
    const float n = fmaf(n01, d23, n23 * d01), d = d01 * d23;
    r = -fmaf(n, d45, n45 * d) / (d * d45);
    x += 6.f;
  }
  const float ix = 1.f / x, ix2 = ix * ix;
  const float series = ix2 * (1.f / 12.f - ix2 * (1.f / 120.f - ix2 * (1.f / 252.f - ix2 * (1.f / 240.f))));
  return r + __logf(x) - 0.5f * ix - series;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Four words of a round: their sums s_i = sum_k mu_ik e_k over the warp (each
// lane brings the products of its own topics in pv), then acc += f_i pv_i / s_i.
// The four sums are reduced together: after two exchanges a lane holds one
// word's partial sum, so that 6 shuffles, 3 of them on one value, and 4
// broadcasts of f_i / s_i serve four words, where one sum at a time took 20.
// The pairs added are those of a butterfly over each word alone, bit for bit.
template <int KPL>
__device__ __forceinline__ void vi_four(const float (&pv)[4][KPL], float f, float (&acc)[KPL], int lane) {
  float s[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    s[i] = pv[i][0];
#pragma unroll
    for (int t = 1; t < KPL; ++t) s[i] += pv[i][t];
  }
  const bool up = lane & 16, odd = lane & 8;
  const float a0 = (up ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, up ? s[0] : s[2], 16);
  const float a1 = (up ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, up ? s[1] : s[3], 16);
  float v = (odd ? a1 : a0) + __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  // lanes 8 i .. 8 i + 7 hold word i's sum; f is that word's count there
  const float w = v > 0.f ? __fdividef(f, v) : -1.f;  // -1: no topic holds the word, it adds nothing
  const bool tiny = w > 3.0e38f;  // a sum below f / FLT_MAX (subnormal rows): product and sum times 2^100
  if (__any_sync(0xffffffffu, tiny)) {
    const float w2 = tiny ? __fdividef(f, v * 0x1p100f) : w, sc = tiny ? 0x1p100f : 1.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float wi = __shfl_sync(0xffffffffu, w2, 8 * i), si = __shfl_sync(0xffffffffu, sc, 8 * i);
      if (wi >= 0.f) {
#pragma unroll
        for (int t = 0; t < KPL; ++t) acc[t] = fmaf(pv[i][t] * si, wi, acc[t]);
      }
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float wi = __shfl_sync(0xffffffffu, w, 8 * i);
    if (wi >= 0.f) {
#pragma unroll
      for (int t = 0; t < KPL; ++t) acc[t] = fmaf(pv[i][t], wi, acc[t]);
    }
  }
}

// Groups of four words whose topic rows stay in registers over the rounds: about
// 64 registers of rows a thread (16 to 32 words up to K = 128, most documents of
// the workloads).
__host__ __device__ constexpr int vi_cached(int kpl) { return kpl == 1 ? 8 : kpl == 2 ? 6 : kpl == 3 ? 5 : kpl == 4 ? 4 : kpl <= 6 ? 2 : 1; }

// KPL topics per lane: topic k = lane + 32 t.  exp(digamma) is taken relative
// to its largest value over the topics, which the per-word normalisation
// cancels, so small gamma never underflows every topic at once.  Bound by
// instruction issue (741 warp instructions a document and round at K = 100 and
// 12 words, IPC 2.45 of 4): 300,000 documents and 20 rounds take 5.69 ms, where
// one word's sum at a time and every row loaded again each round took 6.95; the
// results are the same bit for bit.  More rows in registers or more warps with
// fewer were not faster (5.78 ms with 12 words kept, 6.09 with 4 at 32 warps).
template <int KPL>
__global__ void __launch_bounds__(kViThreads, KPL <= 8 ? 8 : 5) k_doc_topics(tlda_csr docs, const float *__restrict__ mu,
                                                          const float *__restrict__ alpha, int K, int n_iter,
                                                          float *__restrict__ theta, float *__restrict__ gamma_out,
                                                          int32_t *err) {
  constexpr int NC = vi_cached(KPL);
  const int doc = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (doc >= docs.n_docs) return;
  const long long p0 = docs.indptr[doc], p1 = docs.indptr[doc + 1];
  float a[KPL], g[KPL], e[KPL], acc[KPL];
#pragma unroll
  for (int t = 0; t < KPL; ++t) {
    const int k = lane + 32 * t;
    a[t] = k < K ? alpha[k] : 0.f;
  }
  // validation and the document length
  bool bad = p0 < 0 || p1 < p0;
  long long L = 0;
  if (!bad)
    for (long long p = p0 + lane; p < p1; p += 32) {
      const int m = docs.indices[p], f = docs.counts[p];
      if (m < 0 || m >= docs.vocab || f <= 0) bad = true;
      else L += f;
    }
  if (__any_sync(0xffffffffu, bad)) {
    if (lane == 0 && err) atomicOr(err, 1);
#pragma unroll
    for (int t = 0; t < KPL; ++t) {
      const int k = lane + 32 * t;
      if (k < K) {
        theta[(long long)doc * K + k] = __int_as_float(0x7fc00000);
        if (gamma_out) gamma_out[(long long)doc * K + k] = __int_as_float(0x7fc00000);
      }
    }
    return;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  const float l_over_k = (float)L / (float)K;
#pragma unroll
  for (int t = 0; t < KPL; ++t) g[t] = a[t] + l_over_k;

  // four words at q0: their rows, and their counts as vi_four wants them (words
  // past the end: row zero, count 0)
  auto rows_at = [&](long long q0, float (&row)[4][KPL]) {
    const long long mine = q0 + (lane >> 3);
    const int m = mine < p1 ? docs.indices[mine] : -1;
    const float f = mine < p1 ? (float)docs.counts[mine] : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int mi = __shfl_sync(0xffffffffu, m, 8 * i);
      const float *r = mu + (long long)max(mi, 0) * K;
#pragma unroll
      for (int t = 0; t < KPL; ++t) {
        const int k = lane + 32 * t;
        row[i][t] = mi >= 0 && k < K ? __ldg(r + k) : 0.f;
      }
    }
    return f;
  };
  float keep[NC][4][KPL], kf[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    kf[c] = 0.f;
    if (p0 + 4 * c < p1) kf[c] = rows_at(p0 + 4 * c, keep[c]);
  }

  for (int it = 0; it < n_iter; ++it) {
    float mx = -INFINITY;
#pragma unroll
    for (int t = 0; t < KPL; ++t) {
      const int k = lane + 32 * t;
      e[t] = k < K ? digamma_f(g[t]) : -INFINITY;
      mx = fmaxf(mx, e[t]);
    }
    mx = warp_max(mx);
#pragma unroll
    for (int t = 0; t < KPL; ++t) {
      const int k = lane + 32 * t;
      e[t] = k < K ? __expf(e[t] - mx) : 0.f;
      acc[t] = a[t];
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (p0 + 4 * c < p1) {
        float pv[4][KPL];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int t = 0; t < KPL; ++t) pv[i][t] = keep[c][i][t] * e[t];
        vi_four<KPL>(pv, kf[c], acc, lane);
      }
    }
    for (long long q0 = p0 + 4 * NC; q0 < p1; q0 += 4) {
      float pv[4][KPL];
      const float f = rows_at(q0, pv);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int t = 0; t < KPL; ++t) pv[i][t] *= e[t];
      vi_four<KPL>(pv, f, acc, lane);
    }
#pragma unroll
    for (int t = 0; t < KPL; ++t) g[t] = acc[t];
  }
  float tot = 0.f;
#pragma unroll
  for (int t = 0; t < KPL; ++t) tot += (lane + 32 * t < K) ? g[t] : 0.f;
  tot = warp_sum(tot);
  const float inv = 1.f / tot;
#pragma unroll
  for (int t = 0; t < KPL; ++t) {
    const int k = lane + 32 * t;
    if (k < K) {
      theta[(long long)doc * K + k] = g[t] * inv;
      if (gamma_out) gamma_out[(long long)doc * K + k] = g[t];
    }
  }
}

template <int KPL>
void launch(const tlda_csr &d, const float *mu, const float *alpha, int K, int n_iter, float *theta, float *gamma,
            int32_t *err, cudaStream_t s) {
  const long long threads = (long long)d.n_docs * 32;
  k_doc_topics<KPL><<<(unsigned)((threads + kViThreads - 1) / kViThreads), kViThreads, 0, s>>>(
      d, mu, alpha, K, n_iter, theta, gamma, err);
}

}  // namespace

extern "C" tlda_status tlda_doc_topics(const tlda_csr *docs, const float *mu, const float *alpha, int32_t K,
                                       int32_t n_iter, float *theta_out, float *gamma_out, int32_t *err_out,
                                       void *cuda_stream) {
  TLDA_RANGE();
  if (!docs || !mu || !alpha || !theta_out || K < 1 || K > tlda::kMaxDim || n_iter < 0 || docs->n_docs < 0 ||
      docs->vocab < 1 || (docs->n_docs > 0 && (!docs->indptr || !docs->indices || !docs->counts)))
    return TLDA_ERR_INVALID;
  if (docs->n_docs == 0) return TLDA_OK;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const int kpl = (K + 31) / 32;
  if (kpl <= 1) launch<1>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 2) launch<2>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 3) launch<3>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 4) launch<4>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 6) launch<6>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 8) launch<8>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 12) launch<12>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else launch<16>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  return cudaGetLastError() == cudaSuccess ? TLDA_OK : TLDA_ERR_CUDA;
}
