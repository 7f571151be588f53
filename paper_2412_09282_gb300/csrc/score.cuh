// Device helpers of the code search shared by the encode passes and the coupled sweep: codeword
// terms, fp32 score bounds and exact scores in fp32 pairs.
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace crvq {

constexpr float kU = 5.9604645e-08f;    // 2^-24

// Error-bound multiplier: about twice the worst-case FMA-chain analysis (<= 37 + 2 n_fixed).
__host__ __device__ inline float bound_mult(int n_terms) { return 64.f + 4.f * n_terms; }

__device__ __forceinline__ void load_vec(const float* p, float v[kD]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  const float4 b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

__device__ __forceinline__ bool code_ok(int32_t k, int32_t K, unsigned* err) {
  if (k < 0 || k >= K) {
    raise_error(err, ERRBIT_INDEX);
    return false;
  }
  return true;
}

// Codeword terms of the score and of its bound: n = c^T H c (fp32, two FMA chains),
// na = |c|^T |H| |c|, l1 = ||c||_1.
__device__ __forceinline__ void codeword_terms(const float c[kD], const float* H, float& n,
                                               float& na, float& l1) {
  n = 0.f;
  na = 0.f;
  l1 = 0.f;
#pragma unroll
  for (int a = 0; a < kD; ++a) {
    float u = 0.f, ua = 0.f;
#pragma unroll
    for (int b = 0; b < kD; ++b) {
      u = fmaf(H[a * kD + b], c[b], u);
      ua = fmaf(fabsf(H[a * kD + b]), fabsf(c[b]), ua);
    }
    n = fmaf(c[a], u, n);
    na = fmaf(fabsf(c[a]), ua, na);
    l1 += fabsf(c[a]);
  }
}

// fp32 lower / upper bounds s_k -+ Et_k of the score of codeword k from its terms t = (n, Na,
// L1) (codeword_terms): s_k = n + sum_p m2q_p c_p, Et_k = u C (Na + 2 Pmax L1). Any
// evaluation covered by the same error analysis is a valid bound; the fallback needs no more.
__device__ __forceinline__ float low_from(float n, float na, float l1, const float c[kD],
                                          const float m2q[kD], float nbeta, float cmul) {
  float s = fmaf(-kU * cmul, na, n);
#pragma unroll
  for (int p = 0; p < kD; ++p) s = fmaf(m2q[p], c[p], s);
  return fmaf(nbeta, l1, s);
}

__device__ __forceinline__ float up_from(float n, float na, float l1, const float c[kD],
                                         const float m2q[kD], float pmax, float cmul) {
  float s = fmaf(kU * cmul, na, n);
#pragma unroll
  for (int p = 0; p < kD; ++p) s = fmaf(m2q[p], c[p], s);
  return fmaf(2.f * kU * cmul * pmax, l1, s);
}

// Exact scoring in unevaluated fp32 pairs ("double-float"): GB300's fp64 pipe is a small
// fraction of its fp32 rate, so the few decisions that the certified bounds leave open are
// settled with error-free transformations (Knuth's TwoSum, the FMA-based TwoProduct) on the
// fp32 pipe instead. The residual r = t - sum of the fixed codewords is held as rh + rl (exactly for
// one codeword, to 2^-48 of the terms for more); the err (r - c)^T H (r - c) comes out within a few 2^-48
// of |r - c|^T |H| |r - c|: coarser than fp64's 2^-53, far finer than any margin that the data
// determine. TwoProduct is exact above about 2^-102.
namespace dfl {

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// (rh + rl) = t - sum of the fixed codebooks' codewords covering g (codebook order).
__device__ __forceinline__ void target(const SetView& set, const CbList& cbs, int n_fixed,
                                       int64_t i, int64_t g, float rh[kD], float rl[kD],
                                       unsigned* err) {
  load_vec(set.T + i * set.ldT + g * kD, rh);
#pragma unroll
  for (int j = 0; j < kD; ++j) rl[j] = 0.f;
  for (int s = 0; s < n_fixed; ++s) {
    const CbView& cb = cbs.cb[s];
    if (g >= cb.G_cov) continue;
    const int32_t k = cb.codes[i * cb.ld + g];
    if (!code_ok(k, cb.K, err)) continue;
    float c[kD];
    load_vec(cb.C + (int64_t)k * kD, c);
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      float sj, ej;
      two_sum(rh[j], -c[j], sj, ej);
      rh[j] = sj;
      rl[j] = __fadd_rn(rl[j], ej);
    }
  }
}

// err = (r - c)^T H (r - c) as a normalised pair (eh, el), r = rh + rl. NORM: also where r and c cancel
// to a difference below the rounding of the terms that r is left over from (dl would be the larger
// part, and the products keep only its high one).
template <bool NORM = false>
__device__ __forceinline__ void quad_err(const float rh[kD], const float rl[kD],
                                         const float c[kD], const float* H, float& eh,
                                         float& el) {
  float dh[kD], dl[kD];
#pragma unroll
  for (int j = 0; j < kD; ++j) {
    float e;
    two_sum(rh[j], -c[j], dh[j], e);
    dl[j] = __fadd_rn(rl[j], e);
    if (NORM) two_sum(dh[j], dl[j], dh[j], dl[j]);
  }
  float yh[kD], yl[kD];
#pragma unroll
  for (int b = 0; b < kD; ++b) yh[b] = yl[b] = 0.f;
#pragma unroll
  for (int a = 0; a < kD; ++a)
#pragma unroll
    for (int b = 0; b < kD; ++b) {
      const float h = H[a * kD + b];
      const float p = __fmul_rn(dh[a], h);
      const float pe = __fmaf_rn(dh[a], h, -p);  // dh h = p + pe exactly
      float s, t;
      two_sum(yh[b], p, s, t);
      yh[b] = s;
      yl[b] = __fadd_rn(yl[b], __fadd_rn(t, __fmaf_rn(dl[a], h, pe)));
    }
  float sh = 0.f, sl = 0.f;
#pragma unroll
  for (int b = 0; b < kD; ++b) {
    const float p = __fmul_rn(dh[b], yh[b]);
    const float pe = __fmaf_rn(dh[b], yh[b], -p);
    float s, t;
    two_sum(sh, p, s, t);
    sh = s;
    sl = __fadd_rn(sl, __fadd_rn(t, __fmaf_rn(dh[b], yl[b], __fmaf_rn(dl[b], yh[b], pe))));
  }
  eh = __fadd_rn(sh, sl);
  el = __fsub_rn(sl, __fsub_rn(eh, sh));
}

__device__ __forceinline__ bool less(float ah, float al, int ak, float bh, float bl, int bk) {
  return ah < bh || (ah == bh && (al < bl || (al == bl && ak < bk)));
}

}  // namespace dfl

}  // namespace crvq
