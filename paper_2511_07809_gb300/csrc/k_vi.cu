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

// W words of a round (1, 2 or 4): their sums s_i = sum_k mu_ik e_k over the warp
// (each lane brings the products of its own topics in pv), then acc += f_i pv_i / s_i.
// The sums are reduced together: an exchange halves the words that a lane sums,
// so that 6 shuffles, 3 of them on one value, and 4 broadcasts of f_i / s_i serve
// four words, where one sum at a time took 20.  The pairs added are those of a
// butterfly over each word alone, bit for bit.
template <int KPL, int W>
__device__ __forceinline__ void vi_words(const float (&pv)[W][KPL], float f, float (&acc)[KPL], int lane) {
  constexpr int P = 32 / W;  // lanes P i .. P i + P - 1 end with word i's sum; f is that word's count there
  float s[W];
#pragma unroll
  for (int i = 0; i < W; ++i) {
    s[i] = pv[i][0];
#pragma unroll
    for (int t = 1; t < KPL; ++t) s[i] += pv[i][t];
  }
#pragma unroll
  for (int n = W / 2, o = 16; n > 0; n >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < n; ++i)
      s[i] = (up ? s[i + n] : s[i]) + __shfl_xor_sync(0xffffffffu, up ? s[i] : s[i + n], o);
  }
  float v = s[0];
#pragma unroll
  for (int o = P / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const float w = v > 0.f ? __fdividef(f, v) : -1.f;  // -1: no topic holds the word, it adds nothing
  const bool tiny = w > 3.0e38f;  // a sum below f / FLT_MAX (subnormal rows): product and sum times 2^100
  if (__any_sync(0xffffffffu, tiny)) {
    const float w2 = tiny ? __fdividef(f, v * 0x1p100f) : w, sc = tiny ? 0x1p100f : 1.f;
#pragma unroll
    for (int i = 0; i < W; ++i) {
      const float wi = __shfl_sync(0xffffffffu, w2, P * i), si = __shfl_sync(0xffffffffu, sc, P * i);
      if (wi >= 0.f) {
#pragma unroll
        for (int t = 0; t < KPL; ++t) acc[t] = fmaf(pv[i][t] * si, wi, acc[t]);
      }
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < W; ++i) {
    const float wi = W > 1 ? __shfl_sync(0xffffffffu, w, P * i) : w;
    if (wi >= 0.f) {
#pragma unroll
      for (int t = 0; t < KPL; ++t) acc[t] = fmaf(pv[i][t], wi, acc[t]);
    }
  }
}

// How KPL topics a lane are worked: W words reduced together, the rows of the
// first NC W words kept in registers over the rounds, and as many blocks an SM as
// the registers are bounded for.  Measured (10 rounds, V = 3000; one word at a
// time before, in us): warps in flight hide the row gathers better than kept rows,
// except where a row is one register.
//   K = 20, 49 words, 30000 documents     778 -> 508   (nothing kept, 24 blocks: 547)
//   K = 50, 49 words, 30000 documents     963 -> 643   (2 kept groups, 16 blocks: 666)
//   K = 100, 12 words, 50000 documents    671 -> 558   (4 kept groups, 8 blocks: 604)
//   K = 123, 49 words, 18557 documents    888 -> 658   (4 kept groups, 8 blocks: 923)
//   K = 150, 45 words, 18000 documents   1059 -> 747   (2 kept groups, 8 blocks: 1357)
//   K = 180, 45 words, 18000 documents   1222 -> 849   (24 warps an SM in place of 36: 1175)
//   K = 200, 12 words, 20000 documents    528 -> 452   (four words: 456 at best)
//   K = 300, 50 words, 10000 documents   1840 -> 1268  (two words: 1559, four: 1933)
struct ViShape {
  int W, NC, blocks;
};
__host__ __device__ constexpr ViShape vi_shape(int kpl) {
  return kpl <= 1   ? ViShape{4, 4, 16}
         : kpl <= 2 ? ViShape{4, 0, 20}
         : kpl <= 6 ? ViShape{4, 0, 18}
         : kpl <= 7 ? ViShape{2, 0, 16}
         : kpl <= 8 ? ViShape{1, 0, 16}
         : kpl <= 12 ? ViShape{1, 0, 14}
                     : ViShape{1, 0, 10};
}

// KPL topics per lane: topic k = lane + 32 t.  exp(digamma) is taken relative
// to its largest value over the topics, which the per-word normalisation
// cancels, so small gamma never underflows every topic at once.  Bound by
// instruction issue and by the L1/L2 latency of the row gathers: K = 100,
// V = 20000, 100,000 documents of 12 words, 20 rounds take 1.97 ms, where one
// word's sum at a time took 2.40; the results are the same bit for bit.
template <int KPL>
__global__ void __launch_bounds__(kViThreads, vi_shape(KPL).blocks) k_doc_topics(tlda_csr docs, const float *__restrict__ mu,
                                                          const float *__restrict__ alpha, int K, int n_iter,
                                                          float *__restrict__ theta, float *__restrict__ gamma_out,
                                                          int32_t *err) {
  constexpr int NC = vi_shape(KPL).NC, W = vi_shape(KPL).W, P = 32 / W;
  const int doc = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (doc >= docs.n_docs) return;
  const long long p0 = docs.indptr[doc], p1 = docs.indptr[doc + 1];
  float g[KPL], e[KPL], acc[KPL];
  auto prior = [&](int t) { return lane + 32 * t < K ? __ldg(alpha + lane + 32 * t) : 0.f; };
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
  for (int t = 0; t < KPL; ++t) g[t] = prior(t) + l_over_k;

  // a word and its count for each lane from q0 on (past the end: row zero, count 0)
  auto word_at = [&](long long q0, int &m, float &f) {
    m = q0 + lane < p1 ? docs.indices[q0 + lane] : -1;
    f = q0 + lane < p1 ? (float)docs.counts[q0 + lane] : 0.f;
  };
  // the rows of the words that lanes c .. c + W - 1 hold
  auto rows_of = [&](int m, int c, float (&row)[W][KPL]) {
#pragma unroll
    for (int i = 0; i < W; ++i) {
      const int mi = __shfl_sync(0xffffffffu, m, c + i);
      const float *r = mu + (long long)max(mi, 0) * K;
#pragma unroll
      for (int t = 0; t < KPL; ++t) {
        const int k = lane + 32 * t;
        row[i][t] = mi >= 0 && k < K ? __ldg(r + k) : 0.f;
      }
    }
  };
  float keep[NC ? NC : 1][W][KPL], kf[NC ? NC : 1], tf = 0.f;
  int tm = -1;
  word_at(p0, tm, tf);
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    kf[c] = __shfl_sync(0xffffffffu, tf, W * c + lane / P);  // as vi_words wants them
    if (p0 + W * c < p1) rows_of(tm, W * c, keep[c]);
  }
  if (p0 + W * NC < p1) word_at(p0 + W * NC, tm, tf);  // the words after these, requested once

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
      acc[t] = prior(t);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (p0 + W * c < p1) {
        float pv[W][KPL];
#pragma unroll
        for (int i = 0; i < W; ++i)
#pragma unroll
          for (int t = 0; t < KPL; ++t) pv[i][t] = keep[c][i][t] * e[t];
        vi_words<KPL, W>(pv, kf[c], acc, lane);
      }
    }
    int m = tm;
    float f = tf;
    for (long long q0 = p0 + W * NC; q0 < p1; q0 += 32) {
      if (q0 > p0 + W * NC) word_at(q0, m, f);
      const int n = (int)min((long long)32, p1 - q0);
      for (int c = 0; c < n; c += W) {
        float pv[W][KPL];
        rows_of(m, c, pv);
        const float fc = __shfl_sync(0xffffffffu, f, c + lane / P);
#pragma unroll
        for (int i = 0; i < W; ++i)
#pragma unroll
          for (int t = 0; t < KPL; ++t) pv[i][t] *= e[t];
        vi_words<KPL, W>(pv, fc, acc, lane);
      }
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
  else if (kpl <= 5) launch<5>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 6) launch<6>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 7) launch<7>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 8) launch<8>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else if (kpl <= 12) launch<12>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  else launch<16>(*docs, mu, alpha, K, n_iter, theta_out, gamma_out, err_out, s);
  return cudaGetLastError() == cudaSuccess ? TLDA_OK : TLDA_ERR_CUDA;
}
