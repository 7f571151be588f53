// Least-squares codebook update (k-means update step; Alg. 1 FineTuneCodebook in its
// closed-form reading). For codebook `which` with all others fixed, codeword k solves
//   A_k c_k = b_k,  A_k = sum_g cnt[g][k] H_g,  b_k = sum_{v in cluster k} H_{g_v} tau_v,
//   tau_v = t_v - sum over the other covering codebooks of C[code].
//
// Deterministic by construction, with no sort and no float atomics: cnt[g][k] are integer
// counts, b_k is accumulated in 64-bit fixed point (stats.cuh), A_k is summed as fp32 pairs in
// a fixed order (partial sums over fixed slices of the groups, added in slice order), and the
// 8 x 8 system is solved by an fp32 Cholesky factor with iterative refinement whose residual
// is formed in fp32 pairs (to 2^-40 of the solution), in one kernel. GB300's fp64 pipe is a
// small fraction of its fp32 rate and a dependent fp64 operation costs about 180 cycles, so
// none of this arithmetic runs in fp64. The Lloyd encode pass (encode.cu) accumulates the
// same statistics for the codes it writes.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "stats.cuh"

namespace crvq {

namespace {

// The maxima behind the fixed-point scale, and the scale (stats_merge_scale).
__global__ void __launch_bounds__(256)
maxabs_kernel(SetView set, CbList cbs, int which, StatsView st, int64_t n_members, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const int64_t G_cov = st.G_cov;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * blockDim.x;
  float tm = 0.f;
  const int64_t nv = set.M * G_cov;
  for (int64_t v = tid; v < nv; v += nth) {
    const int64_t i = v / G_cov, g = v % G_cov;
    const float4* t = reinterpret_cast<const float4*>(set.T + i * set.ldT + g * kD);
    const float4 a = t[0], b = t[1];
    tm = max_keep_nan(tm, max_keep_nan(max_keep_nan(fabsf(a.x), fabsf(a.y)),
                                       max_keep_nan(fabsf(a.z), fabsf(a.w))));
    tm = max_keep_nan(tm, max_keep_nan(max_keep_nan(fabsf(b.x), fabsf(b.y)),
                                       max_keep_nan(fabsf(b.z), fabsf(b.w))));
  }
  float hm = 0.f;
  for (int64_t r = tid; r < G_cov * kD; r += nth) {
    const float* h = set.Hb + r * kD;
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < kD; ++j) s += fabsf(h[j]);  // a NaN entry makes the sum NaN
    hm = max_keep_nan(hm, s);
  }
  stats_merge_scale(st, cbs, which, tm, hm, n_members, err);
}

// Statistics of every covered vector from its current code, up to 1024 codewords. CTA (x, y): the four
// adjacent groups of quads y, y + gridDim.y, ..., rows x, x + gridDim.x, ... of each, thread = (row,
// group): four lanes read a row's 128 bytes. The CTA sums its counts (per group) and fixed-point
// terms in shared memory (planes of KS entries, KS >= K) and adds them to the global sums once. A term
// (|v| < 2^30) enters shared memory as v = 2^15 vh + vl (0 <= vl < 2^15) in two 32-bit sums (native 32-bit
// atomics): exact, as accumulate_grid gives a CTA fewer than 2^16 vectors of a quad. Integer sums:
// the order is immaterial.
// Bound: load latency and the shared atomics. (With a group per CTA a warp's 32-byte reads lay in 32
// lines: 251 us per codebook of a 28672 x 8192 layer, now 206; k-means step 160 -> 156 us.)
// 257 to 1024 codewords take 80 KB instead of 20, which still leaves two CTAs per SM. Straight to the
// global sums, as larger codebooks go, the few addresses of a small codebook are contended: 12000 x
// 512 vectors took 1.39 ms with 300 codewords and 0.70 with 1024, now 0.117 and 0.142; 64 x 8 vectors,
// the smallest measured, lose 1 to 3 us of 9 to zeroing and flushing.
constexpr int kSmemStatsK = 256, kSmemStatsKMax = 1024;
constexpr int kAccRows = 2;
constexpr int kAccGroups = 4;

constexpr size_t acc_smem(int KS) { return (size_t)KS * (2 * kD + kAccGroups) * sizeof(int); }

template <int KS>
__global__ void __launch_bounds__(256)
accumulate_stats_kernel(SetView set, CbList cbs, int which, StatsView st, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  // [component][vh, vl][code]: lanes of a warp adding one component hit spread banks
  extern __shared__ __align__(16) int s_b32[];
  int* s_cnt = s_b32 + kD * 2 * KS;  // [group of the quad][code]
  const CbView cw = cbs.cb[which];
  const float sscale = stats_scale_f(st);
  const int gq = threadIdx.x % kAccGroups;
  for (int64_t g0 = (int64_t)blockIdx.y * kAccGroups; g0 < cw.G_cov;
       g0 += (int64_t)gridDim.y * kAccGroups) {
    __syncthreads();  // the previous quad's flush has read the sums
    for (int e = threadIdx.x * 4; e < (2 * kD + kAccGroups) * KS; e += blockDim.x * 4)
      *reinterpret_cast<int4*>(s_b32 + e) = make_int4(0, 0, 0, 0);
    __syncthreads();
    const int64_t g = g0 + gq;
    if (g < cw.G_cov) {
      // the group's H block in registers: read once, not 64 loads per vector
      float H[kD * kD];
#pragma unroll
      for (int e = 0; e < kD * kD; e += 4) {
        const float4 h = __ldg(reinterpret_cast<const float4*>(set.Hb + g * kD * kD + e));
        H[e] = h.x;
        H[e + 1] = h.y;
        H[e + 2] = h.z;
        H[e + 3] = h.w;
      }
      // kAccRows rows per step, their codes and vectors loaded before any is used
      const int64_t stride = (int64_t)gridDim.x * (blockDim.x / kAccGroups);
      for (int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kAccGroups; i0 < set.M;
           i0 += kAccRows * stride) {
        int32_t k[kAccRows];
        float tau[kAccRows][kD];
#pragma unroll
        for (int u = 0; u < kAccRows; ++u) {
          const int64_t i = i0 + u * stride;
          k[u] = i < set.M ? cw.codes[i * cw.ld + g] : 0;
          if (i < set.M) stats_target(set, cbs, which, i, g, tau[u], err);
        }
#pragma unroll
        for (int u = 0; u < kAccRows; ++u) {
          if (i0 + u * stride >= set.M) break;
          if (k[u] < 0 || k[u] >= cw.K) {
            raise_error(err, ERRBIT_INDEX);
            continue;
          }
          float q[kD];
          stats_htau(H, tau[u], q);
          atomicAdd(&s_cnt[gq * KS + k[u]], 1);
#pragma unroll
          for (int j = 0; j < kD; ++j) {
            const long long v = fix_rn_small(q[j], sscale);
            atomicAdd(&s_b32[(2 * j) * KS + k[u]], (int)(v >> 15));
            atomicAdd(&s_b32[(2 * j + 1) * KS + k[u]], (int)(v & 0x7fff));
          }
        }
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < cw.K; k += blockDim.x) {
      int all = 0;
#pragma unroll
      for (int q = 0; q < kAccGroups; ++q) {
        const int c = s_cnt[q * KS + k];
        if (c != 0) atomicAdd(&st.cnt[(g0 + q) * st.K + k], c);
        all += c;
      }
      if (all == 0) continue;
#pragma unroll
      for (int j = 0; j < kD; ++j) {
        const long long v =
            (long long)s_b32[(2 * j) * KS + k] * 32768 + s_b32[(2 * j + 1) * KS + k];
        atomicAdd(reinterpret_cast<unsigned long long*>(&st.bacc[(int64_t)k * kD + j]),
                  (unsigned long long)v);
      }
    }
  }
}

// The same for larger codebooks: every vector's terms straight to the global sums. CTA (x, y): groups y,
// y + gridDim.y, ..., thread = row. Bound: latency of the atomics, so it wants many warps: H is read
// per vector (35 registers; with four groups per CTA and H in registers, two CTAs per SM, 12000 x 512
// vectors and 300 codewords took 2.2 ms instead of 1.4).
__global__ void __launch_bounds__(256)
accumulate_global_kernel(SetView set, CbList cbs, int which, StatsView st, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const CbView cw = cbs.cb[which];
  const float sscale = stats_scale_f(st);
  for (int64_t g = blockIdx.y; g < cw.G_cov; g += gridDim.y)
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < set.M;
         i += (int64_t)gridDim.x * blockDim.x) {
      const int32_t k = cw.codes[i * cw.ld + g];
      if (k < 0 || k >= cw.K) {
        raise_error(err, ERRBIT_INDEX);
        continue;
      }
      float tau[kD], q[kD];
      stats_target(set, cbs, which, i, g, tau, err);
      stats_htau(set.Hb + g * kD * kD, tau, q);
      stats_add(st, sscale, g, k, q);
    }
}

// Grid of accumulate_stats_kernel: one column of CTAs per quad of groups, enough of them for about 4
// per SM overall with at least 128 rows each (two per thread), and fewer than 2^16 vectors per
// CTA and quad (the 32-bit shared sums).
dim3 accumulate_grid(int64_t M, int64_t G_cov, int nsm) {
  const int64_t quads = std::max<int64_t>(ceil_div(G_cov, kAccGroups), 1);
  const int64_t want = std::max<int64_t>(1, ceil_div(4 * (int64_t)nsm, quads));
  const int64_t rows_x = std::max<int64_t>(
      ceil_div(M, 65000 / kAccGroups),
      std::max<int64_t>(1, std::min<int64_t>(want, ceil_div(M, 128))));
  return dim3((unsigned)rows_x, (unsigned)std::min<int64_t>(quads, 65535));
}

// Accumulates the statistics of codebook `which` over its M * G_cov > 0 covered vectors.
crvq_status launch_accumulate(const SetView& set, const CbList& cbs, int which, const StatsView& st,
                              unsigned* err, cudaStream_t stream) {
  const CbView& cw = cbs.cb[which];
  const int nsm = sm_count();
  const dim3 grid = accumulate_grid(set.M, cw.G_cov, nsm);
  if (cw.K <= kSmemStatsK) {
    CRVQ_CUDA(launch_pdl(accumulate_stats_kernel<kSmemStatsK>, grid, dim3(256), acc_smem(kSmemStatsK),
                         stream, set, cbs, which, st, err));
  } else if (cw.K <= kSmemStatsKMax) {
    CRVQ_TRY(smem_limit((const void*)accumulate_stats_kernel<kSmemStatsKMax>,
                        acc_smem(kSmemStatsKMax)));
    CRVQ_CUDA(launch_pdl(accumulate_stats_kernel<kSmemStatsKMax>, grid, dim3(256),
                         acc_smem(kSmemStatsKMax), stream, set, cbs, which, st, err));
  } else {
    const int64_t x = std::min<int64_t>(ceil_div(4 * (int64_t)nsm, cw.G_cov), ceil_div(set.M, 1024));
    CRVQ_CUDA(launch_pdl(accumulate_global_kernel,
                         dim3((unsigned)x, (unsigned)std::min<int64_t>(cw.G_cov, 65535)), dim3(256), 0,
                         stream, set, cbs, which, st, err));
  }
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

// fp32 Cholesky factor of the packed lower triangle (false unless every pivot is positive)
// with the reciprocals of its diagonal, and the solve L L^T x = b with them: 8 divisions per
// factor, none per solve (the refinement absorbs the rounding of the reciprocals).
__device__ inline bool chol8_f32(const float A[36], float L[36], float inv[kD]) {
  int q = 0;
#pragma unroll
  for (int r = 0; r < kD; ++r)
#pragma unroll
    for (int c = 0; c <= r; ++c, ++q) {
      float s = A[q];
#pragma unroll
      for (int m = 0; m < c; ++m) s = fmaf(-L[r * (r + 1) / 2 + m], L[c * (c + 1) / 2 + m], s);
      if (r == c) {
        if (!(s > 0.f)) return false;
        L[q] = sqrtf(s);
        inv[r] = 1.f / L[q];
      } else {
        L[q] = s * inv[c];
      }
    }
  return true;
}

__device__ inline void chol8_solve_f32(const float L[36], const float inv[kD], const float b[kD],
                                       float x[kD]) {
  float y[kD];
#pragma unroll
  for (int r = 0; r < kD; ++r) {
    float s = b[r];
#pragma unroll
    for (int m = 0; m < r; ++m) s = fmaf(-L[r * (r + 1) / 2 + m], y[m], s);
    y[r] = s * inv[r];
  }
#pragma unroll
  for (int r = kD - 1; r >= 0; --r) {
    float s = y[r];
#pragma unroll
    for (int m = r + 1; m < kD; ++m) s = fmaf(-L[m * (m + 1) / 2 + r], x[m], s);
    x[r] = s * inv[r];
  }
}

__device__ __forceinline__ void pair_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// Solves A x = b with A (packed lower triangle) and b given as unevaluated fp32 pairs
// (hi + lo), by iterative refinement around an fp32 Cholesky factor: each step forms the
// residual r = b - A x in fp32 pairs (every product split exactly by an FMA, TwoSum
// accumulation, about 2^-44 relative), solves L L^T dx = r in fp32 and adds dx to x, which is
// kept as a pair, until the correction is below 2^-40 of x (each step gains about
// -log2(cond(A) u_32) bits) or after 12 steps. No fp64 arithmetic: a dependent fp64 operation
// costs about 180 cycles on this part. One warp solves one system: the residual, two thirds of
// the arithmetic, is a row per lane (lanes 0-7; the others repeat row 7's work), everything else
// runs redundantly on every lane. Each row's operations and their order are those of a single
// thread, so the result does not depend on the split. Returns false when A has no fp32
// Cholesky factor.
__device__ bool solve8_pairs_warp(const float* __restrict__ Ah, const float* __restrict__ Al,
                                  const float bh[kD], const float bl[kD], float x_out[kD]) {
  const int lane = threadIdx.x & 31, row = min(lane, kD - 1);
  float Lf[36], inv[kD];
  {
    float Af[36];
#pragma unroll
    for (int e = 0; e < 36; ++e) Af[e] = __fadd_rn(Ah[e], Al[e]);
    if (!chol8_f32(Af, Lf, inv)) return false;
  }
  // this lane's row of A and entry of b
  float ah[kD], al[kD], rbh = 0.f, rbl = 0.f;
#pragma unroll
  for (int c = 0; c < kD; ++c) {
    const int q = row >= c ? row * (row + 1) / 2 + c : c * (c + 1) / 2 + row;
    ah[c] = Ah[q];
    al[c] = Al[q];
    if (c == row) {
      rbh = bh[c];
      rbl = bl[c];
    }
  }
  float bf[kD], xh[kD], xl[kD];
#pragma unroll
  for (int j = 0; j < kD; ++j) {
    bf[j] = __fadd_rn(bh[j], bl[j]);
    xl[j] = 0.f;
  }
  chol8_solve_f32(Lf, inv, bf, xh);
  for (int it = 0; it < 12; ++it) {
    float h = rbh, l = rbl;
#pragma unroll
    for (int c = 0; c < kD; ++c) {
      const float p = __fmul_rn(ah[c], xh[c]);
      const float pe = __fmaf_rn(ah[c], xh[c], -p);  // Ah xh = p + pe exactly
      const float cross = __fmaf_rn(ah[c], xl[c], __fmul_rn(al[c], xh[c]));
      float sum, t;
      pair_two_sum(h, -p, sum, t);
      h = sum;
      l = __fadd_rn(l, __fsub_rn(t, __fadd_rn(pe, cross)));
    }
    const float mine = __fadd_rn(h, l);
    float rf[kD];
#pragma unroll
    for (int r = 0; r < kD; ++r) rf[r] = __shfl_sync(0xffffffffu, mine, r);
    float dx[kD];
    chol8_solve_f32(Lf, inv, rf, dx);
    float xm = 0.f, dm = 0.f;
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      float sum, t;
      pair_two_sum(xh[j], dx[j], sum, t);
      const float lo = __fadd_rn(xl[j], t);
      xh[j] = __fadd_rn(sum, lo);                      // renormalise the pair
      xl[j] = __fsub_rn(lo, __fsub_rn(xh[j], sum));
      xm = fmaxf(xm, fabsf(xh[j]));
      dm = fmaxf(dm, fabsf(dx[j]));
    }
    if (dm <= 9.094947e-13f * xm) break;  // 2^-40 (the same on every lane)
  }
#pragma unroll
  for (int j = 0; j < kD; ++j) x_out[j] = __fadd_rn(xh[j], xl[j]);
  return true;
}

// The fp64 Cholesky solve, for a matrix without an fp32 factor (cond(A) beyond fp32; rare).
__device__ __noinline__ bool solve8_f64(const float* Ah, const float* Al, const float bh[kD],
                                        const float bl[kD], float out[kD]) {
  double A[36], b[kD], x[kD];
  for (int v = 0; v < 36; ++v) A[v] = (double)Ah[v] + (double)Al[v];
  for (int j = 0; j < kD; ++j) b[j] = (double)bh[j] + (double)bl[j];
  if (!cholesky_solve8(A, b, x)) return false;
  for (int j = 0; j < kD; ++j) out[j] = (float)x[j];
  return true;
}

// b_j = bacc_j / 2^sexp as an fp32 pair: the int64 fixed-point sum split into three exact
// 24-bit pieces, added by TwoSum, scaled by a power of two.
__device__ __forceinline__ void fixed_to_pair(long long v, int sexp, float& h, float& l) {
  const int a2 = (int)(v >> 48);                    // |a2| < 2^15
  const int a1 = (int)((v >> 24) & 0xffffff);
  const int a0 = (int)(v & 0xffffff);
  float s, t;
  pair_two_sum((float)a2 * 281474976710656.f, (float)a1 * 16777216.f, s, t);  // 2^48, 2^24
  float s2, t2;
  pair_two_sum(s, (float)a0, s2, t2);
  h = ldexpf(s2, -sexp);
  l = ldexpf(__fadd_rn(t, t2), -sexp);
}

// The least-squares solve of every codeword, one kernel. CTA = NC codewords; thread = (entry
// e of A_k's packed lower triangle or the count, slice of the groups). Each thread sums
// cnt[g][k] * H_g[e] over its slice as an unevaluated fp32 pair for each of the CTA's codewords
// (every product is split exactly: cnt < 2^24; TwoSum for the high part), so no fp64 arithmetic
// runs per group and an H entry is read once for all NC codewords; the slices are added in a fixed
// order as fp32 pairs, and then a warp per codeword solves A_k c_k = b_k (b_k from the fixed point)
// by Cholesky with refinement in fp32 pairs. The fixed assignment and order make the result
// identical on every run. Codewords without members keep their old value.
// Bound: latency (0.4 MB per launch). As two kernels, the solve with one thread per codeword, a 512 x
// 512 layer (64 groups) took 5.3 + 8.0 us per Lloyd iteration; one kernel saves 4.8 us of that, and
// nothing at 512 groups, where the sums' own work is the larger part; two slices per thread took 19 us
// there, one takes 14. NC is the smallest of 2, 4 and 8 that makes a single wave (one CTA per SM), 8 beyond
// that: with 2 always, two of a CTA's 18 warps solved while the next CTAs waited (371 groups: 65536
// codewords 2.32 ms, now 1.17; 4096: 141 us, now 83; 1024: 43 us, now 25; 256 keep 2: 16 us, 24 with 8).
constexpr int kSolveSlices = 16;  // groups split 16 ways: short dependent chains per thread
constexpr int kSumThreads = kSolveSlices * kNA;  // 592

template <int NC>
__global__ void __launch_bounds__(kSumThreads)
stats_solve_kernel(const float* __restrict__ Hb, StatsView st, const float* C_old, float* C_out,
                   int32_t* __restrict__ counts_out, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  __shared__ float part_h[NC][kSolveSlices][kNA], part_l[NC][kSolveSlices][kNA];
  __shared__ float sAh[NC][kNA], sAl[NC][kNA];
  const int tid = threadIdx.x;
  const int sl = tid / kNA;
  const int e = tid % kNA;
  const int K = st.K;
  const int k0 = blockIdx.x * NC;
  const int nk = min(NC, K - k0);
  // entry e of the packed lower triangle: row r, column c (c <= r); e = 36 is the count
  int r = 0;
  while ((r + 1) * (r + 2) / 2 <= e && r < kD - 1) ++r;
  const int c = e - r * (r + 1) / 2;
  const int hoff = r * kD + c;
  float hi[NC], lo[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) hi[q] = lo[q] = 0.f;
  // slice sl: gper groups, in group order
  const int64_t gper = (st.G_cov + kSolveSlices - 1) / kSolveSlices;
  const int64_t g0 = sl * gper, g1 = min(st.G_cov, g0 + gper);
  constexpr int kBatch = 8;  // groups whose loads are in flight together; no branches
  for (int64_t gb = 0; gb < gper; gb += kBatch) {
    float fc[kBatch][NC], h[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int64_t g = g0 + gb + u;
      const bool in = g < g1;
#pragma unroll
      for (int q = 0; q < NC; ++q)  // exact: counts stay below 2^24
        fc[u][q] = in && q < nk ? (float)st.cnt[g * K + k0 + q] : 0.f;
      h[u] = in ? (e < 36 ? __ldg(Hb + g * kD * kD + hoff) : 1.f) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const float p = __fmul_rn(fc[u][q], h[u]);
        const float pe = __fmaf_rn(fc[u][q], h[u], -p);  // fc h = p + pe exactly
        float sum, t;
        pair_two_sum(hi[q], p, sum, t);
        hi[q] = sum;
        lo[q] = __fadd_rn(lo[q], __fadd_rn(t, pe));
      }
  }
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    part_h[q][sl][e] = hi[q];
    part_l[q][sl][e] = lo[q];
  }
  __syncthreads();
  // Every thread has read its counts: clear them, so that the statistics are zero for the next
  // accumulation (the Lloyd loop needs no memset between iterations).
  for (int64_t v = tid; v < st.G_cov * nk; v += kSumThreads)
    st.cnt[(v / nk) * K + k0 + v % nk] = 0;
  // Slices are merged per entry by one thread in fp32 pairs (TwoSum of the high parts, low parts
  // added), in slice order.
  for (int v = tid; v < NC * kNA; v += kSumThreads) {
    const int q = v / kNA, eq = v % kNA;
    float h = part_h[q][0][eq], l = part_l[q][0][eq];
#pragma unroll
    for (int s2 = 1; s2 < kSolveSlices; ++s2) {
      float sum, t;
      pair_two_sum(h, part_h[q][s2][eq], sum, t);
      h = sum;
      l = __fadd_rn(l, __fadd_rn(t, part_l[q][s2][eq]));
    }
    sAh[q][eq] = h;
    sAl[q][eq] = l;
  }
  __syncthreads();
  const int kq = tid >> 5, k = k0 + kq;  // warp kq solves codeword k
  if (kq >= nk) return;
  const float* Ah = sAh[kq];
  const float* Al = sAl[kq];
  // the count: an exact integer held by the pair
  const int64_t count = (int64_t)__float2int_rn(Ah[36]) + (int64_t)__float2int_rn(Al[36]);
  if (counts_out && (tid & 31) == 0) counts_out[k] = (int32_t)count;
  bool keep = count == 0;
  float out[kD];
  if (!keep) {
    const int sexp = stats_scale_exp(*st.scale);
    float bh[kD], bl[kD];
#pragma unroll
    for (int j = 0; j < kD; ++j) fixed_to_pair(st.bacc[(int64_t)k * kD + j], sexp, bh[j], bl[j]);
    __syncwarp();
    if ((tid & 31) == 0)
#pragma unroll
      for (int j = 0; j < kD; ++j) st.bacc[(int64_t)k * kD + j] = 0;  // read: clear (see above)
    if (!solve8_pairs_warp(Ah, Al, bh, bl, out)) {
      if (!solve8_f64(Ah, Al, bh, bl, out)) {
        if ((tid & 31) == 0) raise_error(err, ERRBIT_NUMERIC);
        keep = true;
      }
    }
  }
  if ((tid & 31) != 0) return;
#pragma unroll
  for (int j = 0; j < kD; ++j) C_out[(int64_t)k * kD + j] = keep ? C_old[(int64_t)k * kD + j] : out[j];
}

crvq_status launch_solve_kernels(const float* Hb, const StatsView& st, const float* C_old,
                                 float* C_out, int32_t* counts, unsigned* err,
                                 cudaStream_t stream) {
  ProfScope ps("update_solve", stream, (double)st.K);
  auto run = [&](auto nc) -> cudaError_t {
    constexpr int NC = decltype(nc)::value;
    return launch_pdl(stats_solve_kernel<NC>, dim3((unsigned)ceil_div(st.K, NC)), dim3(kSumThreads), 0,
                      stream, Hb, st, C_old, C_out, counts, err);
  };
  const int nsm = sm_count();
  CRVQ_CUDA(st.K <= 2 * nsm   ? run(std::integral_constant<int, 2>{})
            : st.K <= 4 * nsm ? run(std::integral_constant<int, 4>{})
                              : run(std::integral_constant<int, 8>{}));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

}  // namespace

crvq_status stats_alloc(Scratch& mem, int64_t G_cov, int K, StatsView* st, cudaStream_t s) {
  CRVQ_TRY(mem.alloc(stats_layout(G_cov, K).total, s));
  stats_bind(mem.as<char>(), G_cov, K, st);
  return stats_zero(*st, s);
}

crvq_status stats_zero(const StatsView& st, cudaStream_t s) {
  const StatsLayout L = stats_layout(st.G_cov, st.K);
  CRVQ_CUDA(cudaMemsetAsync(st.cnt, 0, L.total, s));
  return CRVQ_OK;
}

static crvq_status launch_maxabs(const SetView& set, const CbList& cbs, int which,
                                 const StatsView& st, unsigned* err, cudaStream_t stream) {
  const int64_t n = set.M * cbs.cb[which].G_cov;
  ProfScope ps("update_bound", stream, (double)n * kD * 4.0);
  CRVQ_CUDA(launch_pdl(maxabs_kernel, dim3((unsigned)std::max<int64_t>(1,
                       std::min<int64_t>(ceil_div(n, 256), 4 * sm_count()))), dim3(256), 0, stream,
                       set, cbs, which, st, std::max<int64_t>(1, n), err));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

crvq_status launch_stats_prepare(const SetView& set, const CbList& cbs, int which,
                                 const StatsView& st, cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  return launch_maxabs(set, cbs, which, st, err, stream);
}

crvq_status launch_stats_solve(const SetView& set, const StatsView& st, const float* C_old,
                               float* C_out, int32_t* counts, cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  return launch_solve_kernels(set.Hb, st, C_old, C_out, counts, err, stream);
}

crvq_status launch_update_codebook(const SetView& set, const CbList& cbs, int which,
                                   float* C_out, int32_t* counts, cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  const CbView& cw = cbs.cb[which];
  const int64_t n = set.M * cw.G_cov;
  Scratch mem;
  StatsView st;
  CRVQ_TRY(stats_alloc(mem, cw.G_cov, cw.K, &st, stream));
  CRVQ_TRY(launch_stats_prepare(set, cbs, which, st, stream));
  if (n > 0) {
    ProfScope ps("update_accumulate", stream, (double)n);
    CRVQ_TRY(launch_accumulate(set, cbs, which, st, err, stream));
  }
  return launch_stats_solve(set, st, cw.C, C_out, counts, stream);
}

}  // namespace crvq

namespace crvq {

// The update of launch_update_codebook on caller-provided scratch (no allocation): `scratch`
// (256-byte aligned, `bytes` long) holds cnt | bacc | scale + maxima, and `err` is the error
// word the kernels report to. Returns CRVQ_ERR_UNSUPPORTED when the statistics of this
// codebook do not fit in `bytes`.
// The size limit counts K * 296 bytes beyond what the kernels use (the documented limit).
size_t update_scratch_bytes(int64_t G_cov, int K) {
  return stats_layout(G_cov, K).total + align_up((size_t)K * kNA * sizeof(float2), 256);
}

crvq_status launch_update_codebook_on(const SetView& set, const CbList& cbs, int which,
                                      float* C_out, int32_t* counts, void* scratch,
                                      size_t bytes, unsigned* err, cudaStream_t stream) {
  const CbView& cw = cbs.cb[which];
  const int64_t n = set.M * cw.G_cov;
  const size_t need = update_scratch_bytes(cw.G_cov, cw.K);
  if (need > bytes)
    return fail(CRVQ_ERR_UNSUPPORTED,
                "statistics of this codebook need %zu bytes of scratch, the limit is %zu "
                "(G_cov * K * 4 + K * 64 + 256 + K * 296 bytes, each part 256-byte aligned)",
                need, bytes);
  const StatsLayout L = stats_layout(cw.G_cov, cw.K);
  StatsView st;
  stats_bind(scratch, cw.G_cov, cw.K, &st);
  // The scratch keeps the previous call's contents: clear counts, sums and maxima.
  CRVQ_CUDA(cudaMemsetAsync(scratch, 0, L.total, stream));
  CRVQ_TRY(launch_maxabs(set, cbs, which, st, err, stream));
  if (n > 0) CRVQ_TRY(launch_accumulate(set, cbs, which, st, err, stream));
  return launch_solve_kernels(set.Hb, st, cw.C, C_out, counts, err, stream);
}

}  // namespace crvq
