// Vector x codeword score contraction with fused top-B selection (Sec. 3.1 Eq. (2)-(3);
// Alg. 1 VectorQuant and BeamSearchOptimize), and the k-means initial codebook draw.
//
// Score of target r against codeword c for a vector of group g:
//   err(r, c) = (r - c)^T H_g (r - c) = r^T H_g r + n_g(c) - 2 (H_g r) . c,  n_g(c) = c^T H_g c.
// The fast pass evaluates the expanded form in fp32 (8 FMAs per pair; the codewords, their
// group norms and L1 norms staged in shared memory). Every fp32 score s_k comes with an
// a-priori bound on its rounding error,
//   E_k <= Et_k = u C (Na_k + 2 Pmax L1_k),   u = 2^-24,
//   Na_k = |c_k|^T |H_g| |c_k|,  L1_k = ||c_k||_1,  Pmax = max_p sum_j |H_pj| (|t_j| + sum_f |c_f,j|),
// and the pass ranks the lower bounds low_k = s_k - Et_k, keeping the best two. The arg-min j
// is certified when low_2nd - low_j > 2 Et_j: every other codeword's exact score is then larger
// than j's. Otherwise the vector is open: the codewords with low_k <= low_j + 2 Et_j (the exact
// arg-min is among them) are decided among in fp32 pairs (score.cuh). Codes therefore equal the fp64
// arg-min (ties to the smaller index) except for ties below the pairs' resolution, a few 2^-48 of
// |r - c|^T |H| |r - c|. Beam stages use the same bounds on a sorted top-(B+1) list.
#include <algorithm>
#include <cstdlib>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "kernels.h"
#include "score.cuh"
#include "stats.cuh"
#include "tc_ops.cuh"

namespace crvq {

namespace {

constexpr int kThreads = 128;
constexpr int kChunk = 256;             // codewords staged per shared-memory chunk
struct FlagList {
  int64_t* vec;      // vector index within the launch range (i * G_range + (g - g_begin))
  float* thr;        // decision threshold (fast-pass value units)
  unsigned* count;
  int64_t cap;
  unsigned long long* total;  // optional running total of flagged vectors
};

// --------------------------------------------------------------------------- device helpers
// fp32 target r = t - sum of the fixed codebooks covering g (codebook order), and the
// magnitude bound a_j = |t_j| + sum |c_fixed,j| of every term that went into r.
__device__ __forceinline__ void target32(const SetView& set, const CbList& cbs, int n_fixed,
                                         int64_t i, int64_t g, float r[kD], float a[kD],
                                         unsigned* err) {
  load_vec(set.T + i * set.ldT + g * kD, r);
#pragma unroll
  for (int j = 0; j < kD; ++j) a[j] = fabsf(r[j]);
  for (int s = 0; s < n_fixed; ++s) {
    const CbView& cb = cbs.cb[s];
    if (g >= cb.G_cov) continue;
    const int32_t k = cb.codes[i * cb.ld + g];
    if (!code_ok(k, cb.K, err)) continue;
    float c[kD];
    load_vec(cb.C + (int64_t)k * kD, c);
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      r[j] -= c[j];
      a[j] += fabsf(c[j]);
    }
  }
}

// fp64 target (the fixed reconstruction subtracted in fp64, codebook order).
__device__ void target64(const SetView& set, const CbList& cbs, int n_fixed, int64_t i,
                         int64_t g, double r[kD], unsigned* err) {
  const float* t = set.T + i * set.ldT + g * kD;
#pragma unroll
  for (int j = 0; j < kD; ++j) r[j] = (double)t[j];
  for (int s = 0; s < n_fixed; ++s) {
    const CbView& cb = cbs.cb[s];
    if (g >= cb.G_cov) continue;
    const int32_t k = cb.codes[i * cb.ld + g];
    if (!code_ok(k, cb.K, err)) continue;
    const float* c = cb.C + (int64_t)k * kD;
#pragma unroll
    for (int j = 0; j < kD; ++j) r[j] -= (double)c[j];
  }
}

// (r - c)^T H (r - c) in fp64; H row-major d x d (fp32); c fp32 or null.
__device__ double quad_err64(const double r[kD], const float* c, const float* H) {
  double dlt[kD];
#pragma unroll
  for (int j = 0; j < kD; ++j) dlt[j] = r[j] - (c ? (double)c[j] : 0.0);
  double e = 0.0;
#pragma unroll
  for (int b = 0; b < kD; ++b) {
    double hb = 0.0;
#pragma unroll
    for (int a2 = 0; a2 < kD; ++a2) hb += dlt[a2] * (double)H[a2 * kD + b];
    e += hb * dlt[b];
  }
  return e;
}

// Vector terms: m2q = -2 H r (the row FMA chains of stats_htau), Pmax = max_p (|H| a)_p.
__device__ __forceinline__ void vector_terms(const float r[kD], const float a[kD],
                                             const float* H, float m2q[kD], float& pmax) {
  pmax = 0.f;
#pragma unroll
  for (int p = 0; p < kD; ++p) {
    float q = 0.f, pa = 0.f;
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      q = fmaf(H[p * kD + j], r[j], q);
      pa = fmaf(fabsf(H[p * kD + j]), a[j], pa);
    }
    m2q[p] = -2.f * q;
    pmax = fmaxf(pmax, pa);
  }
}

// vector_terms plus rr = r^T (H r) and Ra = a^T (|H| a), each row of H read once as two
// float4 (H 16-byte aligned): the same FMA chains, so the same values as computing them apart.
__device__ __forceinline__ void vector_terms_rr(const float r[kD], const float a[kD],
                                                const float* H, float m2q[kD], float& pmax,
                                                float& rr, float& ra) {
  pmax = 0.f;
  rr = 0.f;
  ra = 0.f;
#pragma unroll
  for (int p = 0; p < kD; ++p) {
    const float4 h0 = *reinterpret_cast<const float4*>(H + p * kD);
    const float4 h1 = *reinterpret_cast<const float4*>(H + p * kD + 4);
    const float hr[kD] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
    float q = 0.f, pa = 0.f;
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      q = fmaf(hr[j], r[j], q);
      pa = fmaf(fabsf(hr[j]), a[j], pa);
    }
    m2q[p] = -2.f * q;
    pmax = fmaxf(pmax, pa);
    rr = fmaf(r[p], q, rr);
    ra = fmaf(a[p], pa, ra);
  }
}

// Stage the codewords [k0, k0 + nk): sC = c, sNL = (n - u C Na, ||c||_1) (the lower-bound
// offset of the codeword part and its L1 norm), sNa = Na.
__device__ __forceinline__ void stage_chunk(const float* __restrict__ C, int k0, int nk,
                                            const float* sH, float cmul, float* sC, float2* sNL,
                                            float* sNa) {
  for (int k = threadIdx.x; k < nk; k += blockDim.x) {
    float c[kD];
    load_vec(C + (int64_t)(k0 + k) * kD, c);
    float n, na, l1;
    codeword_terms(c, sH, n, na, l1);
    *reinterpret_cast<float4*>(sC + k * kD) = make_float4(c[0], c[1], c[2], c[3]);
    *reinterpret_cast<float4*>(sC + k * kD + 4) = make_float4(c[4], c[5], c[6], c[7]);
    sNL[k] = make_float2(n - kU * cmul * na, l1);
    sNa[k] = na;
  }
}

// --------------------------------------------------------------------------- arg-min pass on
// the tensor cores. The whole certified lower bound is one dot product of length 32:
//   D[v][k] = sum_p q_vp c_kp + n'_k + beta_v L1_k + off_v = low_k(v) + off_v,
//   q = -2 H_g r, n' = n - u C Na, beta = -2 u C Pmax, off >= r^T H r + bound (so D >= 0),
// with every term split into tf32 hi + lo (3xTF32: hi*hi + hi*lo + lo*hi):
//   A row (vector):   [q_hi x8 | q_hi x8 | q_lo x8 | 1 1 | beta_hi beta_hi beta_lo | off_hi off_lo | 0]
//   B row (codeword): [c_hi x8 | c_lo x8 | c_hi x8 | n'_hi n'_lo | L1_hi L1_lo L1_hi | 1 1 | 0]
// One tcgen05.mma M = 128 vectors x N = 128 codewords x K = 8, four per chunk (K = 32), fp32
// accumulator in tensor memory. The epilogue takes minima of the non-negative scores as integer minima
// of their bit patterns, along the columns in two ways, so that the smallest of each name the winner's
// column (argmin_small_kernel, argmin_tc_kernel). The certificate is that of the fp32 pass, with the bound
// multiplier raised to cover the tensor-core products and accumulation (about 2^-22 per split product
// and fp32 accumulation over 32 terms); rows without it are decided in fp32 pairs.
namespace tcenc {

constexpr int kRows = 128;        // vectors per row tile (TMEM lanes)
constexpr int kK = 32;            // tf32 columns per row
constexpr int kATile = kRows * kK * 4;   // 16 KB
constexpr float kCmul = 256.f;           // bound multiplier (about twice the analysis)

__device__ __forceinline__ uint32_t koff(int r, int k) {
  return (uint32_t)(((r >> 3) * (kK / 4) + (k >> 2)) * 128 + (r & 7) * 16 + (k & 3) * 4);
}

// Writes the 32 tf32 values v[0..31] of row r (hi parts given as fp32 values).
__device__ __forceinline__ void put_row(char* tile, int r, const uint32_t v[kK]) {
#pragma unroll
  for (int q = 0; q < kK / 4; ++q)
    *reinterpret_cast<uint4*>(tile + koff(r, 4 * q)) =
        make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}

__device__ __forceinline__ void split(float x, uint32_t& hi, uint32_t& lo) {
  hi = tc::to_tf32(x);
  lo = tc::to_tf32(x - __uint_as_float(hi));
}

}  // namespace tcenc

// Row of the B operand for codeword kk of C (K codewords): [c_hi | c_lo | c_hi | n'_hi n'_lo |
// L1_hi L1_lo L1_hi | 1 1 | 0]; padding rows (kk >= K) score +1e30.
// t = (n, Na, L1) of the codeword (codeword_terms; zeros for padding).
__device__ __forceinline__ void build_b_row(const float* __restrict__ C, int K, int kk,
                                            const float* H, float uc, uint32_t row[tcenc::kK],
                                            float t[3]) {
  using namespace tcenc;
  t[0] = t[1] = t[2] = 0.f;
  if (kk < K) {
    float cv[kD], n, na, l1;
    load_vec(C + (int64_t)kk * kD, cv);
    codeword_terms(cv, H, n, na, l1);
    t[0] = n;
    t[1] = na;
    t[2] = l1;
#pragma unroll
    for (int p = 0; p < kD; ++p) {
      uint32_t hh, ll;
      split(cv[p], hh, ll);
      row[p] = hh;
      row[8 + p] = ll;
      row[16 + p] = hh;
    }
    split(n - uc * na, row[24], row[25]);
    split(l1, row[26], row[27]);
    row[28] = row[26];
  } else {
#pragma unroll
    for (int p = 0; p < 24; ++p) row[p] = 0u;
    row[24] = __float_as_uint(1e30f);
    row[25] = 0u;
    row[26] = row[27] = row[28] = 0u;
  }
  row[29] = row[30] = __float_as_uint(1.f);
  row[31] = 0u;
}

// cbmax[0] = max_k ||c_k||_1 (raised by 1e-6 relative), cbmax[1] = max_k,j |c_kj|: one CTA
// of any size up to 1024 threads (maxima are order-free).
__device__ void cbmax_block(const float* __restrict__ C, int K, float* __restrict__ cbmax) {
  __shared__ float r1[32], r2[32];
  float l1m = 0.f, cm = 0.f;
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    float c[kD];
    load_vec(C + (int64_t)k * kD, c);
    float l1 = 0.f;
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      l1 += fabsf(c[j]);
      cm = fmaxf(cm, fabsf(c[j]));
    }
    l1m = fmaxf(l1m, l1);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    l1m = fmaxf(l1m, __shfl_xor_sync(0xffffffffu, l1m, off));
    cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, off));
  }
  if ((threadIdx.x & 31) == 0) {
    r1[threadIdx.x >> 5] = l1m;
    r2[threadIdx.x >> 5] = cm;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)((blockDim.x + 31) >> 5); ++w) {
      l1m = fmaxf(l1m, r1[w]);
      cm = fmaxf(cm, r2[w]);
    }
    cbmax[0] = l1m * (1.f + 1e-6f);
    cbmax[1] = cm;
  }
}

constexpr int kTcCols = 128;                     // codewords per chunk (MMA N)
constexpr int kTcBTile = kTcCols * tcenc::kK * 4;  // 16 KB

// B operand images of the codebook for the groups g_begin + blockIdx.y: block (g, chunk) holds 128
// rows in the canonical shared-memory layout, ready for a bulk copy. terms[g_rel K + k] = (n, Na, L1, 0)
// of codeword k in the group (codeword_terms). A CTA stays in its group, whose H block it reads once.
__global__ void __launch_bounds__(128)
prep_b_kernel(SetView set, int64_t g_begin, const float* __restrict__ C, int K, int nchunk, float uc,
              char* __restrict__ out, float4* __restrict__ terms, float* __restrict__ cbmax,
              unsigned* __restrict__ flag_count) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  // The flag list of the beam stage that follows starts empty. The previous stage's fallback, which
  // read the count, completed before the wait above returned.
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *flag_count = 0u;
  if (blockIdx.x == gridDim.x - 1) {  // the last column of CTAs: the codebook maxima (its first)
    if (blockIdx.y == 0) cbmax_block(C, K, cbmax);
    return;
  }
  const int64_t g = g_begin + blockIdx.y;
  float H[kD * kD];
#pragma unroll
  for (int e = 0; e < kD * kD; e += 4) {
    const float4 h = __ldg(reinterpret_cast<const float4*>(set.Hb + g * kD * kD + e));
    H[e] = h.x;
    H[e + 1] = h.y;
    H[e + 2] = h.z;
    H[e + 3] = h.w;
  }
  for (int chunk = blockIdx.x; chunk < nchunk; chunk += gridDim.x - 1) {
    const int kk = chunk * kTcCols + threadIdx.x;
    uint32_t v[tcenc::kK];
    float tk[3];
    build_b_row(C, K, kk, H, uc, v, tk);
    tcenc::put_row(out + ((int64_t)blockIdx.y * nchunk + chunk) * kTcBTile, threadIdx.x, v);
    if (kk < K) terms[(int64_t)blockIdx.y * K + kk] = make_float4(tk[0], tk[1], tk[2], 0.f);
  }
}

// Grid of prep_b_kernel: about 16 CTAs per SM in all, and the column that takes the maxima.
dim3 prep_b_grid(int64_t G_range, int nchunk, int nsm) {
  const int64_t x = std::max<int64_t>(1, std::min<int64_t>(nchunk, ceil_div(16 * (int64_t)nsm, G_range)));
  return dim3((unsigned)x + 1, (unsigned)G_range);
}

// The same rows for codebooks of more than 256 codewords, in two parts: of a row's 32 values only n'
// depends on the group. A chunk's 128 rows are laid out by four-value columns of 2 KB (kBCol), and column
// 6 (n'_hi n'_lo L1_hi L1_lo) is stored per group: out_g[(g_rel nchunk + chunk) 2 KB]; the others once:
// out[chunk 16 KB], column 6 unused. A group takes 1 MB for 65536 codewords instead of 8, and 128
// groups share a pass instead of 32. K = 65536, 1024 x 11008: 43 passes of (124 us images, 390 us
// arg-min) became 11 of (97 us, 1331 us), 25.2 -> 17.4 ms in all.
constexpr int kBCol = kTcCols * 16;
constexpr int kBGroupCol = 6;

__global__ void __launch_bounds__(128)
prep_b_split_kernel(SetView set, int64_t g_begin, const float* __restrict__ C, int K, int nchunk, float uc,
                    bool first, char* __restrict__ out, char* __restrict__ out_g,
                    float4* __restrict__ terms, float* __restrict__ cbmax,
                    unsigned* __restrict__ flag_count) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  // The open lists of the arg-min pass that follows start empty. The previous pass's exact kernels,
  // which read the counts, completed before the wait above returned.
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 2) flag_count[threadIdx.x] = 0u;
  if (blockIdx.x == gridDim.x - 1) {  // the last column of CTAs: the codebook maxima (its first)
    if (first && blockIdx.y == 0) cbmax_block(C, K, cbmax);
    return;
  }
  const int64_t g = g_begin + blockIdx.y;
  float H[kD * kD];
#pragma unroll
  for (int e = 0; e < kD * kD; e += 4) {
    const float4 h = __ldg(reinterpret_cast<const float4*>(set.Hb + g * kD * kD + e));
    H[e] = h.x;
    H[e + 1] = h.y;
    H[e + 2] = h.z;
    H[e + 3] = h.w;
  }
  for (int chunk = blockIdx.x; chunk < nchunk; chunk += gridDim.x - 1) {
    const int kk = chunk * kTcCols + threadIdx.x;
    uint32_t v[tcenc::kK];
    float tk[3];
    build_b_row(C, K, kk, H, uc, v, tk);
    char* row = out + (int64_t)chunk * kTcBTile + threadIdx.x * 16;
    if (first && blockIdx.y == 0)
#pragma unroll
      for (int q = 0; q < tcenc::kK / 4; ++q)
        if (q != kBGroupCol)
          *reinterpret_cast<uint4*>(row + q * kBCol) =
              make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    constexpr int e = 4 * kBGroupCol;
    *reinterpret_cast<uint4*>(out_g + ((int64_t)blockIdx.y * nchunk + chunk) * kBCol +
                              threadIdx.x * 16) = make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]);
    if (kk < K) terms[(int64_t)blockIdx.y * K + kk] = make_float4(tk[0], tk[1], tk[2], 0.f);
  }
}

// Per-vector terms of the arg-min's A rows that do not change while one codebook's Lloyd
// iterations run (the target, H_g and the fixed codebooks stay put): m2q = -2 H_g r and rr,
// Ra, Pmax (vector_terms_rr of target32), as three planes of M float4 per group,
// rt[(3 g + p) M + i]: p = 0, 1 the two halves of m2q, p = 2 (rr, Ra, Pmax, 0). The arg-min
// pass reads them instead of recomputing them, with bit-identical values.
// With statistics (st.cnt) it also takes the maxima behind their fixed-point scale from the vectors
// it reads, and sets the scale (stats_merge_scale): a pass over the matrix and two launches less per
// codebook fit.
__global__ void __launch_bounds__(128)
row_terms_kernel(SetView set, CbList cbs, int n_fixed, float4* __restrict__ rt, StatsView st,
                 unsigned* err) {
  pdl_trigger();
  pdl_wait();
  const int64_t nvec = set.M * set.G_sub;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * blockDim.x;
  float tm = 0.f;
  for (int64_t v = tid; v < nvec; v += nth) {
    const int64_t g = v / set.M, i = v - g * set.M;
    float rv[kD], a[kD], m2q[kD], pmax, rr, ra;
    target32(set, cbs, n_fixed, i, g, rv, a, err);
    vector_terms_rr(rv, a, set.Hb + g * kD * kD, m2q, pmax, rr, ra);  // H_g 16-byte aligned
    rt[(3 * g) * set.M + i] = make_float4(m2q[0], m2q[1], m2q[2], m2q[3]);
    rt[(3 * g + 1) * set.M + i] = make_float4(m2q[4], m2q[5], m2q[6], m2q[7]);
    rt[(3 * g + 2) * set.M + i] = make_float4(rr, ra, pmax, 0.f);
    float t[kD];
    load_vec(set.T + i * set.ldT + g * kD, t);
#pragma unroll
    for (int j = 0; j < kD; ++j) tm = max_keep_nan(tm, fabsf(t[j]));
  }
  if (!st.cnt) return;
  float hm = 0.f;
  for (int64_t r = tid; r < set.G_sub * kD; r += nth) {
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < kD; ++j) s += fabsf(set.Hb[r * kD + j]);  // a NaN entry makes the sum NaN
    hm = max_keep_nan(hm, s);
  }
  stats_merge_scale(st, cbs, n_fixed, tm, hm, nvec > 0 ? nvec : 1, err);
}

constexpr int kSmallK = 2 * kTcCols;   // codebooks up to this size stay resident in shared memory
constexpr int kTcSmemStatsK = kSmallK;  // and sum their statistics there

// Minimum of 16 non-negative fp32 values by their bit patterns (which order like the values),
// as three-input integer minima.
__device__ __forceinline__ uint32_t min16_bits(const uint32_t* x) {
  const uint32_t a = __vimin3_u32(x[0], x[1], x[2]), b = __vimin3_u32(x[3], x[4], x[5]),
                 c = __vimin3_u32(x[6], x[7], x[8]), d = __vimin3_u32(x[9], x[10], x[11]),
                 e = __vimin3_u32(x[12], x[13], x[14]);
  return min(__vimin3_u32(a, b, c), __vimin3_u32(d, e, x[15]));
}

constexpr int kBlk = 16;  // columns per block of the arg-min sweep

// --------------------------------------------------------------------------- arg-min pass,
// codebooks of at most 256 codewords: bounds, certificate, exact decisions and Lloyd statistics
// in one persistent kernel.
//
// The work is the linear list of (group, pair of 128-row tiles); CTA c takes an equal share of
// it, a run of pairs that touches one group or a few. Per group ("segment") the CTA builds the
// group's B operand itself, a thread per codeword (about 2 k cycles; a separate kernel writing
// images took 8 us per pass and 32 KB of L2 traffic per group and CTA), and then two halves of 128
// threads run independently over alternate tiles, as tile pipelines: A rows, MMA per chunk of 128
// codewords, sweep, certificate, statistics (own A tile, named barrier, mbarrier, 128 accumulator
// columns each). Two CTAs per SM, so four pipelines interleave.
//
// Sweep. A row's 256 scores D form a 16 x 16 grid (block b = column / 16, class e = column % 16).
// Kept are the minimum of every block and of every class, as three-input integer minima of the
// non-negative fp32 bit patterns: 0.5 + 0.5 instructions per score and no per-score index. The
// smallest score is the smallest block minimum and the smallest class minimum, so its block and
// class name its column; the runner-up differs from it in block or class, so it is the second
// smallest block minimum or the second smallest class minimum, exactly. (Keeping the winning block's
// 16 values by selects instead cost 0.6 per score more on the ALU pipe, the busiest one.)
//
// Open rows. When the runner-up is within the bound `top` of the winner the row is open: every
// column whose exact score could be the smallest has D <= top, so its block and its class have
// minima <= top, and the two 16-bit masks of those name all candidates (two to four columns as a
// rule, instead of the whole codebook). They go to a list in shared memory, and after its last tile
// the CTA decides its open rows exactly (dfl, fp32 pairs), eight lanes per row (a warp each when they
// are at most eight). A row that finds the list full is decided at once by its warp. This replaces a
// kernel that gave every open row a warp and scanned the codebook twice (21 us per pass of a 4096 x
// 4096 matrix, 9 us of a 512 x 512).
constexpr int kOpenCap = 256;  // open rows a CTA keeps for its end

struct OpenRow {
  uint32_t i, g;   // row, group (absolute)
  uint32_t masks;  // blocks << 16 | classes
};

constexpr size_t kArgminSmem = 2 * (size_t)tcenc::kATile + 2 * (size_t)kTcBTile +
                               (size_t)kTcSmemStatsK * (kD * 8 + 4) +
                               4 * (size_t)tcenc::kRows * kD * 4 + (size_t)kTcSmemStatsK * 8 +
                               (size_t)kOpenCap * sizeof(OpenRow) + 1024;

// Exact decision of one open row (i, g) by the eight lanes of a quarter warp (all 32 lanes call it; a
// quarter with live = false takes part without writing): the candidates k = cand(0 .. total - 1)
// are scored in fp32 pairs (H: the group's block), the smallest (err, index) wins, its statistics
// are added when requested.
template <class Cand>
__device__ __forceinline__ void decide_open(const SetView& set, const CbList& cbs, int n_fixed,
                                            int s_idx, int64_t i, int64_t g, bool live, int total,
                                            Cand cand, int32_t* __restrict__ out_code,
                                            int64_t out_ld, int64_t out_g0, const StatsView& st,
                                            float sscale, unsigned* err) {
  const CbView& cw = cbs.cb[s_idx];
  const int sub = threadIdx.x & 7;
  const float* H = set.Hb + g * kD * kD;
  float rh[kD], rl[kD];
  dfl::target(set, cbs, n_fixed, i, g, rh, rl, err);
  float bh = INFINITY, bl = 0.f;
  int bk = 0x7fffffff;
  for (int c = sub; c < total; c += 8) {
    const int k = cand(c);
    if (k >= cw.K) continue;  // padding columns
    float cv[kD], eh, el;
    load_vec(cw.C + (int64_t)k * kD, cv);
    dfl::quad_err(rh, rl, cv, H, eh, el);
    if (dfl::less(eh, el, k, bh, bl, bk)) {
      bh = eh;
      bl = el;
      bk = k;
    }
  }
  __syncwarp();
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, bh, off);
    const float ol = __shfl_xor_sync(0xffffffffu, bl, off);
    const int ok = __shfl_xor_sync(0xffffffffu, bk, off);
    if (dfl::less(oh, ol, ok, bh, bl, bk)) {
      bh = oh;
      bl = ol;
      bk = ok;
    }
  }
  if (sub == 0 && live) {
    if (bk == 0x7fffffff) {
      raise_error(err, ERRBIT_NUMERIC);  // no candidate: non-finite scores
    } else {
      if (out_code) out_code[i * out_ld + (g - out_g0)] = bk;
      if (st.cnt) {
        float q[kD];
        stats_htau(H, rh, q);  // rh is the fp32 target (TwoSum's rounded sums)
        stats_add(st, sscale, g, bk, q);
      }
    }
  }
}

// Index of the (n + 1)-th set bit of m.
__device__ __forceinline__ int nth_bit(uint32_t m, int n) {
  for (; n > 0; --n) m &= m - 1u;
  return __ffs(m) - 1;
}

// decide_open of a row of the small-codebook pass: blocks x classes of its masks.
__device__ __forceinline__ void decide_grid(const SetView& set, const CbList& cbs, int n_fixed,
                                            int s_idx, const OpenRow& o, bool live,
                                            int32_t* __restrict__ out_code, int64_t out_ld,
                                            int64_t out_g0, const StatsView& st, float sscale,
                                            unsigned* err) {
  const uint32_t bm = o.masks >> 16, em = o.masks & 0xffffu;
  const int ne = __popc(em);
  decide_open(set, cbs, n_fixed, s_idx, o.i, o.g, live, __popc(bm) * ne,
              [&](int c) { return kBlk * nth_bit(bm, c / ne) + nth_bit(em, c % ne); }, out_code,
              out_ld, out_g0, st, sscale, err);
}

// The smallest value of v[0..N) (w1, at index idx; the first of equal ones) and the second
// smallest (w2, equal to w1 when it occurs twice).
template <int N>
__device__ __forceinline__ void top2(const uint32_t v[N], uint32_t& w1, uint32_t& w2, int& idx) {
  w1 = v[0];
  w2 = 0xffffffffu;
  idx = 0;
#pragma unroll
  for (int e = 1; e < N; ++e) {
    w2 = min(w2, max(w1, v[e]));
    idx = v[e] < w1 ? e : idx;
    w1 = min(w1, v[e]);
  }
}

// Smallest and second smallest of v[0..16) with their low four bits replaced by the index: w1 & 15
// is where the smallest lies, values are known to within 15 units. Two trees of three-input
// minima: in p - w1 - 1 the smallest itself wraps around to the largest. 48 instructions in short
// chains, where the running top-2 with an index (top2) takes 75 in chains of 15; a 28672 x 8192 layer
// went from 83.2 to 82.2 ms, a 512 x 512 one from 1.57 to 1.52 ms.
__device__ __forceinline__ void top2_packed(const uint32_t v[16], uint32_t& w1, uint32_t& w2) {
  uint32_t p[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) p[e] = (v[e] & ~15u) | (uint32_t)e;
  w1 = min16_bits(p);
#pragma unroll
  for (int e = 0; e < 16; ++e) p[e] = p[e] - w1 - 1u;
  w2 = min16_bits(p) + w1 + 1u;
}

template <int N>
__device__ __forceinline__ uint32_t mask_le(const uint32_t v[N], uint32_t top) {
  uint32_t m = 0;
#pragma unroll
  for (int e = 0; e < N; ++e) m |= v[e] <= top ? 1u << e : 0u;
  return m;
}

// Barrier over one half's 128 threads (named barrier 1 + half), with an AND of v.
__device__ __forceinline__ bool half_sync_and(int half, bool v) {
  int r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 q, %1, 0;\n bar.red.and.pred p, %2, 128, q;\n"
      " selp.s32 %0, 1, 0, p;\n}\n"
      : "=r"(r)
      : "r"((int)v), "r"(1 + half)
      : "memory");
  return r != 0;
}

// decide_grid of one row by a whole warp: four candidates at a time, lane b of eight takes column b of
// H (r - c); the same operations in the same order as dfl::quad_err's, so the same err pairs. About
// 260 dependent instructions per four candidates instead of 700: for a CTA with few open rows,
// whose end they are (a Lloyd pass over 512 x 64 vectors 16.7 -> 15.3 us, the codes' stores included).
__device__ __forceinline__ void decide_grid_warp(const SetView& set, const CbList& cbs, int n_fixed,
                                                 int s_idx, const OpenRow& o,
                                                 int32_t* __restrict__ out_code, int64_t out_ld,
                                                 int64_t out_g0, const StatsView& st, float sscale,
                                                 unsigned* err) {
  const CbView& cw = cbs.cb[s_idx];
  const int lane = threadIdx.x & 31, b = lane & 7, base = lane & 24;
  const int64_t i = o.i, g = o.g;
  const uint32_t bm = o.masks >> 16, em = o.masks & 0xffffu;
  const int ne = __popc(em), total = __popc(bm) * ne;
  const float* H = set.Hb + g * kD * kD;
  float hb[kD];  // column b
#pragma unroll
  for (int a = 0; a < kD; ++a) hb[a] = __ldg(H + a * kD + b);
  float rh[kD], rl[kD];
  dfl::target(set, cbs, n_fixed, i, g, rh, rl, err);
  float bh = INFINITY, bl = 0.f;
  int bk = 0x7fffffff;
  for (int c0 = 0; c0 < total; c0 += 4) {
    const int c = c0 + (lane >> 3);
    const int k = c < total ? kBlk * nth_bit(bm, c / ne) + nth_bit(em, c % ne) : cw.K;
    const bool valid = k < cw.K;  // (the others are padding columns)
    float cv[kD], dh[kD], dl[kD], yh = 0.f, yl = 0.f;
    load_vec(cw.C + (int64_t)(valid ? k : 0) * kD, cv);
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      float e;
      dfl::two_sum(rh[j], -cv[j], dh[j], e);
      dl[j] = __fadd_rn(rl[j], e);
    }
#pragma unroll
    for (int a = 0; a < kD; ++a) {
      const float p = __fmul_rn(dh[a], hb[a]);
      const float pe = __fmaf_rn(dh[a], hb[a], -p);  // dh h = p + pe exactly
      float s, t;
      dfl::two_sum(yh, p, s, t);
      yh = s;
      yl = __fadd_rn(yl, __fadd_rn(t, __fmaf_rn(dl[a], hb[a], pe)));
    }
    float sh = 0.f, sl = 0.f;
#pragma unroll
    for (int q = 0; q < kD; ++q) {
      const float qh = __shfl_sync(0xffffffffu, yh, base + q);
      const float ql = __shfl_sync(0xffffffffu, yl, base + q);
      const float p = __fmul_rn(dh[q], qh);
      const float pe = __fmaf_rn(dh[q], qh, -p);
      float s, t;
      dfl::two_sum(sh, p, s, t);
      sh = s;
      sl = __fadd_rn(sl, __fadd_rn(t, __fmaf_rn(dh[q], ql, __fmaf_rn(dl[q], qh, pe))));
    }
    const float eh = __fadd_rn(sh, sl), el = __fsub_rn(sl, __fsub_rn(eh, sh));
    if (valid && dfl::less(eh, el, k, bh, bl, bk)) {
      bh = eh;
      bl = el;
      bk = k;
    }
  }
#pragma unroll
  for (int off = 8; off < 32; off <<= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, bh, off);
    const float ol = __shfl_xor_sync(0xffffffffu, bl, off);
    const int ok = __shfl_xor_sync(0xffffffffu, bk, off);
    if (dfl::less(oh, ol, ok, bh, bl, bk)) {
      bh = oh;
      bl = ol;
      bk = ok;
    }
  }
  if (bk == 0x7fffffff) {
    if (lane == 0) raise_error(err, ERRBIT_NUMERIC);  // no candidate: non-finite scores
    return;
  }
  if (lane == 0 && out_code) out_code[i * out_ld + (g - out_g0)] = bk;
  if (st.cnt && lane < kD) {  // stats_add, a component per lane
    float a = 0.f;
#pragma unroll
    for (int c = 0; c < kD; ++c) a = fmaf(__ldg(H + lane * kD + c), rh[c], a);
    if (lane == 0) atomicAdd(&st.cnt[g * st.K + bk], 1);
    atomicAdd(reinterpret_cast<unsigned long long*>(&st.bacc[(int64_t)bk * kD + lane]),
              (unsigned long long)fix_rn_small(a, sscale));
  }
}

__global__ void __launch_bounds__(256, 2)
argmin_small_kernel(SetView set, int64_t g_begin, int64_t G_range, CbList cbs, int n_fixed,
                    int s_idx, int32_t* __restrict__ out_code, int64_t out_ld, int64_t out_g0,
                    unsigned long long* flag_total, StatsView st,
                    const float4* __restrict__ rowterms, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor below
  using namespace tcenc;
  extern __shared__ __align__(1024) char smem_raw[];
  // 1024-byte aligned base, derived from the shared array (keeps the shared address space)
  char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  char* Atiles = smem;                    // 2 x 16 KB
  char* Bbuf = smem + 2 * kATile;         // 2 x 16 KB
  int* s_b32 = reinterpret_cast<int*>(Bbuf + 2 * kTcBTile);     // [8][2][256] statistics halves
  int* s_cnt = s_b32 + kTcSmemStatsK * kD * 2;                  // [256]
  float* sQ = reinterpret_cast<float*>(s_cnt + kTcSmemStatsK);  // [2][256][8]: H r of a row
  float2* sNaL1 = reinterpret_cast<float2*>(sQ + 4 * kRows * kD);      // [256]
  OpenRow* s_open = reinterpret_cast<OpenRow*>(sNaL1 + kTcSmemStatsK);  // [kOpenCap]
  __shared__ __align__(16) float sH[kD * kD];
  __shared__ __align__(8) uint64_t bar_mma_s[2];
  __shared__ uint32_t tmem_slot;
  __shared__ float s_l1[8], s_cinf[8];
  __shared__ unsigned n_open, s_repeated[8];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int half = tid >> 7, rrow = tid & (kRows - 1);
  char* Atile = Atiles + half * kATile;
  uint64_t& bar_mma = bar_mma_s[half];
  const CbView cw = cbs.cb[s_idx];
  const float cmul = kCmul + 4.f * n_fixed;
  const float uc = kU * cmul;
  const int nchunk = cw.K > kTcCols ? 2 : 1;

  // Before the wait only this block's shared memory is touched.
  if (tid == 0) {
    n_open = 0;
    tc::mbar_init(tc::smem_u32(&bar_mma_s[0]), 1);
    tc::mbar_init(tc::smem_u32(&bar_mma_s[1]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int e = tid; e < kTcSmemStatsK * kD * 2; e += 256) s_b32[e] = 0;
  s_cnt[tid] = 0;
  // Repeated codewords. Only the first of equal ones can be a row's code, so the others get padding
  // columns: scored, they would leave every row nearest to them open with all of them as candidates (a
  // matrix whose vectors are zero by half, where most codewords are zero too: a pass over 4096 x 512
  // vectors took 12.5 ms, now 0.13). Two hash tables (in sQ, not in use yet) keep the smallest codeword of
  // each slot. A repeated one that finds another codeword first in both of its slots goes unnoticed, and
  // costs time only.
  constexpr int kSlots = 1024;
  int* s_slot = reinterpret_cast<int*>(sQ);                             // [2][kSlots]
  uint32_t* s_hash = reinterpret_cast<uint32_t*>(s_slot + 2 * kSlots);  // [256]
  uint32_t hash = 0;
#pragma unroll
  for (int e = 0; e < 2; ++e)
    *reinterpret_cast<int4*>(s_slot + 4 * (tid + 256 * e)) = make_int4(256, 256, 256, 256);
  __syncthreads();
  pdl_wait();
  if (warp == 0) tc::tmem_alloc(&tmem_slot, 2 * kTcCols);
  float cv[kD];
#pragma unroll
  for (int j = 0; j < kD; ++j) cv[j] = 0.f;
  if (tid < cw.K) load_vec(cw.C + (int64_t)tid * kD, cv);
  {  // codebook maxima: max_k ||c_k||_1 (raised by 1e-6 relative) and max |c|
    float l1 = 0.f, cm = 0.f;
    if (tid < cw.K) {
#pragma unroll
      for (int j = 0; j < kD; ++j) {
        l1 += fabsf(cv[j]);
        cm = fmaxf(cm, fabsf(cv[j]));
        hash += __float_as_uint(__fadd_rn(cv[j], 0.f)) * (0x9E3779B1u * (2 * j + 1));  // (-0 as 0)
      }
      hash ^= hash >> 13;
      hash *= 0x85EBCA6Bu;
      atomicMin(&s_slot[hash >> 22], tid);
      atomicMin(&s_slot[kSlots + ((hash >> 12) & (kSlots - 1))], tid);
      s_hash[tid] = hash;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      l1 = fmaxf(l1, __shfl_xor_sync(0xffffffffu, l1, off));
      cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, off));
    }
    if (lane == 0) {
      s_l1[warp] = l1;
      s_cinf[warp] = cm;
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  {
    bool repeated = false;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int first = s_slot[e == 0 ? hash >> 22 : kSlots + ((hash >> 12) & (kSlots - 1))];
      if (first < tid && s_hash[first] == hash && tid < cw.K) {
        float o[kD];
        load_vec(cw.C + (int64_t)first * kD, o);
        bool same = true;
#pragma unroll
        for (int j = 0; j < kD; ++j) same = same && cv[j] == o[j];
        repeated = repeated || same;
      }
    }
    const unsigned rep = __ballot_sync(0xffffffffu, repeated);
    if (lane == 0) s_repeated[warp] = rep;  // (read by its own warp, after the first segment's barrier)
  }
  // this half's accumulator: columns [128 half, 128 half + 128)
  const uint32_t tmem = tmem_slot + (uint32_t)(half * kTcCols);
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const float sscale = st.cnt ? stats_scale_f(st) : 1.f;
  float l1max = 0.f, cinf = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    l1max = fmaxf(l1max, s_l1[w]);
    cinf = fmaxf(cinf, s_cinf[w]);
  }
  l1max *= 1.f + 1e-6f;
  constexpr uint32_t idesc = tc::idesc_tf32(kRows, kTcCols);

  // this CTA's share [p, p_end) of the G_range * pairs_g tile pairs
  const int64_t pairs_g = (set.M + 2 * kRows - 1) / (2 * kRows);
  const int64_t total = G_range * pairs_g;
  int64_t p = total * blockIdx.x / gridDim.x;
  const int64_t p_end = total * (blockIdx.x + 1) / gridDim.x;
  bool ok = true;
  int mma_count = 0;

  while (p < p_end) {
    // one segment: pairs of one group, fewer than 2^16 rows (the 32-bit statistics halves)
    const int64_t grel = p / pairs_g, g = g_begin + grel;
    const int64_t pg = p - grel * pairs_g;  // the segment's first pair within the group
    const int np = (int)min(min(p_end - p, pairs_g - pg), (int64_t)255);
    if (tid < kD * kD) sH[tid] = set.Hb[g * kD * kD + tid];
    __syncthreads();
    {  // B operand of the group: thread = codeword
      uint32_t row[kK];
      float tk[3];
      if (tid < nchunk * kTcCols) {
        build_b_row(cw.C, (s_repeated[warp] >> lane) & 1u ? 0 : cw.K, tid, sH, uc, row, tk);
        put_row(Bbuf + (tid >> 7) * kTcBTile, tid & (kTcCols - 1), row);
        sNaL1[tid] = make_float2(tk[1], tk[2]);
      }
    }
    tc::fence_async_smem();
    __syncthreads();
    // Bound on Na_k over the codebook for this group: (max row sum |H_g|) L1max cinf.
    float hrow = 0.f;
#pragma unroll
    for (int a = 0; a < kD; ++a) {
      float rs = 0.f;
#pragma unroll
      for (int b = 0; b < kD; ++b) rs += fabsf(sH[a * kD + b]);
      hrow = fmaxf(hrow, rs);
    }

    // This thread's terms of row i (row_terms_kernel's planes; zeros past the rows).
    auto load_terms = [&](int64_t i, float4& q0, float4& q1, float4& t2) {
      q0 = q1 = t2 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < set.M) {
        q0 = rowterms[(3 * g) * set.M + i];
        q1 = rowterms[(3 * g + 1) * set.M + i];
        t2 = rowterms[(3 * g + 2) * set.M + i];
      }
    };
    // The A row of row i, from its terms when they are precomputed; H r to sQ[buf].
    auto make_row = [&](int64_t i, const float4& q0, const float4& q1, const float4& t2, int buf,
                        float& pmax, float& off) {
      float m2q[kD], rr, ra;
      if (rowterms) {
        m2q[0] = q0.x; m2q[1] = q0.y; m2q[2] = q0.z; m2q[3] = q0.w;
        m2q[4] = q1.x; m2q[5] = q1.y; m2q[6] = q1.z; m2q[7] = q1.w;
        rr = t2.x;
        ra = t2.y;
        pmax = t2.z;
      } else {
        float rv[kD], a[kD];
        if (i < set.M) {
          target32(set, cbs, n_fixed, i, g, rv, a, err);
        } else {
#pragma unroll
          for (int j = 0; j < kD; ++j) rv[j] = a[j] = 0.f;
        }
        vector_terms_rr(rv, a, sH, m2q, pmax, rr, ra);
      }
      // offset making every D = low + off >= 0, with margins for every rounding involved
      off = (rr + 32.f * kU * ra + 2.f * uc * (hrow * l1max * cinf + 2.f * pmax * l1max)) *
                (1.f + 4.f * uc) + 1e-30f;
      const float beta = -2.f * uc * pmax;
      if (st.cnt) {  // H r of this row, kept for the statistics (-m2q / 2, exact)
        float* q = sQ + (buf * 256 + tid) * kD;
        *reinterpret_cast<float4*>(q) =
            make_float4(-0.5f * m2q[0], -0.5f * m2q[1], -0.5f * m2q[2], -0.5f * m2q[3]);
        *reinterpret_cast<float4*>(q + 4) =
            make_float4(-0.5f * m2q[4], -0.5f * m2q[5], -0.5f * m2q[6], -0.5f * m2q[7]);
      }
      uint32_t row[kK];
#pragma unroll
      for (int q = 0; q < kD; ++q) {
        uint32_t h, l;
        split(m2q[q], h, l);
        row[q] = h;
        row[8 + q] = h;
        row[16 + q] = l;
      }
      const uint32_t one = __float_as_uint(1.f);
      row[24] = one;
      row[25] = one;
      split(beta, row[26], row[28]);
      row[27] = row[26];
      split(off * (1.f - uc), row[29], row[30]);
      row[31] = 0u;
      put_row(Atile, rrow, row);
      tc::fence_async_smem();
    };
    auto issue = [&](int c) {  // chunk c's MMA into this half's accumulator
      if (rrow == 0) {
        tc::tc_fence_after();
        const uint32_t a0 = tc::smem_u32(Atile), b0 = tc::smem_u32(Bbuf + c * kTcBTile);
#pragma unroll
        for (int ks = 0; ks < kK / 8; ++ks)
          tc::mma_tf32(tmem, tc::smem_desc(a0 + ks * 256, 128, (kK / 4) * 128),
                       tc::smem_desc(b0 + ks * 256, 128, (kK / 4) * 128), idesc, ks > 0 ? 1u : 0u);
        tc::mma_commit(tc::smem_u32(&bar_mma));
      }
    };
    auto wait_mma = [&]() -> bool {  // the same answer in the whole warp
      const bool done = tc::mbar_wait(tc::smem_u32(&bar_mma), (uint32_t)(mma_count & 1), err);
      ++mma_count;
      tc::tc_fence_after();
      return __all_sync(0xffffffffu, done);
    };

    // Software pipeline of a half: while a tile's certificate and statistics run, the next tile's
    // first MMA does, and the next tile's terms are loaded before the sweep.
    int64_t i = (pg * 2 + half) * kRows + rrow;
    float pmax, off;
    {
      float4 q0, q1, t2;
      if (rowterms) load_terms(i, q0, q1, t2);
      make_row(i, q0, q1, t2, 0, pmax, off);
    }
    ok = half_sync_and(half, ok);
    if (ok) issue(nchunk - 1);
    for (int t = 0; t < np && ok; ++t) {
      const bool row_ok = i < set.M, more = t + 1 < np;
      const int64_t i_next = i + 2 * kRows;
      float4 q0, q1, t2;
      if (rowterms && more) load_terms(i_next, q0, q1, t2);
      uint32_t mb[kBlk], mc[kBlk];  // block and class minima (fp32 bits)
#pragma unroll
      for (int e = 0; e < kBlk; ++e) mb[e] = mc[e] = 0xffffffffu;
      auto sweep = [&](auto chunk) {
        constexpr int c = decltype(chunk)::value;
#pragma unroll
        for (int rnd = 0; rnd < 2; ++rnd) {
          uint32_t v[64];
          tc::tmem_ld64_wait(trow + 64 * rnd, v);
#pragma unroll
          for (int q = 0; q < 4; ++q) mb[8 * c + 4 * rnd + q] = min16_bits(v + kBlk * q);
#pragma unroll
          for (int e = 0; e < kBlk; ++e) {
            mc[e] = __vimin3_u32(mc[e], v[e], v[kBlk + e]);
            mc[e] = __vimin3_u32(mc[e], v[2 * kBlk + e], v[3 * kBlk + e]);
          }
        }
      };
      ok = wait_mma();
      if (nchunk == 2) {  // chunk 1 first: the last sweep is always chunk 0's
        if (ok) sweep(std::integral_constant<int, 1>{});
        tc::tc_fence_before();
        ok = half_sync_and(half, ok);  // the accumulator has been read; ok uniform in the half
        if (ok) {
          issue(0);
          ok = wait_mma();
        }
      }
      // this tile's MMAs are done with the A tile: the next tile's rows
      float pmax_next = 0.f, off_next = 0.f;
      if (ok && more) make_row(i_next, q0, q1, t2, (t + 1) & 1, pmax_next, off_next);
      if (ok) sweep(std::integral_constant<int, 0>{});
      tc::tc_fence_before();
      ok = half_sync_and(half, ok);  // rows written, accumulator read
      if (!ok) break;
      if (more) issue(nchunk - 1);

      // Certificate, code, open row and statistics of this thread's row.
      bool open = false;
      OpenRow o{};
      if (row_ok) {
        uint32_t w1, w2, x1, x2;
        top2_packed(mb, w1, w2);
        top2_packed(mc, x1, x2);
        const uint32_t s2 = min(w2, x2) & ~15u;
        int j = (int)(w1 & 15u) * kBlk + (int)(x1 & 15u);
        const float k1 = __uint_as_float(w1 | 15u);  // >= the winner's score
        const float k2 = s2 >= 0xfffffff0u ? INFINITY : __uint_as_float(s2);  // <= the others'
        bool cert = false;
        float top = INFINITY;
        if (j < cw.K) {
          const float2 tj = sNaL1[j];
          // D_k <= s_k + off (every k); s_j + off <= D_j + e2 (the winner): no other codeword's
          // exact score reaches s_j when k2 > D_j + e2 (the sum rounded up).
          float e2 = 2.f * uc * (tj.x + 2.f * pmax * tj.y + off);
          top = __fadd_ru(k1, e2);   // >= s_j + off
          cert = cw.K == 1 || k2 > top;
          // (nearly) equal scores: block and class may name different columns; the bound over all
          // codewords
          if (s2 == (w1 & ~15u)) {
            e2 = 2.f * uc * (hrow * l1max * cinf + 2.f * pmax * l1max + off) * 1.0001f;
            top = __fadd_ru(k1, e2);
          }
        } else {
          j = 0;
        }
        if (!cert) {
          open = true;
          const uint32_t tb = __float_as_uint(top) & 0x7fffffffu;
          o.i = (uint32_t)i;
          o.g = (uint32_t)g;
          o.masks = (mask_le<kBlk>(mb, tb) << 16) | mask_le<kBlk>(mc, tb);
        }
        if (out_code) out_code[i * out_ld + (g - out_g0)] = j;
        if (cert && st.cnt) {
          // H r from the prologue (bit-identical to the standalone update's H tau). A term v
          // (|v| < 2^30) enters as v = 2^15 vh + vl, 0 <= vl < 2^15, in two 32-bit sums: exact,
          // since a segment has fewer than 2^16 rows.
          float q[kD];
          load_vec(sQ + ((t & 1) * 256 + tid) * kD, q);
          atomicAdd(&s_cnt[j], 1);
#pragma unroll
          for (int e = 0; e < kD; ++e) {
            const long long v = fix_rn_small(q[e], sscale);
            atomicAdd(&s_b32[(2 * e) * kTcSmemStatsK + j], (int)(v >> 15));
            atomicAdd(&s_b32[(2 * e + 1) * kTcSmemStatsK + j], (int)(v & 0x7fff));
          }
        }
      }
      // open rows: to the list, or decided here when it is full
      bool over = false;
      if (open) {
        const unsigned slot = atomicAdd(&n_open, 1u);
        if (slot < (unsigned)kOpenCap)
          s_open[slot] = o;
        else
          over = true;
      }
      unsigned om = __ballot_sync(0xffffffffu, over);
      while (om) {  // four rows at a time, a quarter warp each
        int src = -1;
        unsigned rest = om;
        for (int q = 0; q < 4 && rest; ++q) {
          if (q == lane >> 3) src = __ffs(rest) - 1;
          rest &= rest - 1u;
        }
        const int from = src < 0 ? __ffs(om) - 1 : src;
        OpenRow w;
        w.i = __shfl_sync(0xffffffffu, o.i, from);
        w.g = __shfl_sync(0xffffffffu, o.g, from);
        w.masks = __shfl_sync(0xffffffffu, o.masks, from);
        decide_grid(set, cbs, n_fixed, s_idx, w, src >= 0, out_code, out_ld, out_g0, st, sscale,
                    err);
        om = rest;
      }
      i = i_next;
      pmax = pmax_next;
      off = off_next;
    }
    ok = __syncthreads_and(ok);  // both halves are done with the group's operand and statistics
    if (st.cnt && tid < cw.K) {  // flush (integer sums: order-free) and clear
      const int c = s_cnt[tid];
      if (c != 0) {
        s_cnt[tid] = 0;
        atomicAdd(&st.cnt[g * st.K + tid], c);
#pragma unroll
        for (int e = 0; e < kD; ++e) {
          int* ph = &s_b32[(2 * e) * kTcSmemStatsK + tid];
          int* pl = &s_b32[(2 * e + 1) * kTcSmemStatsK + tid];
          const long long v = (long long)*ph * 32768 + *pl;
          *ph = 0;
          *pl = 0;
          atomicAdd(reinterpret_cast<unsigned long long*>(&st.bacc[(int64_t)tid * kD + e]),
                    (unsigned long long)v);
        }
      }
    }
    if (!ok) break;
    p += np;
  }
  // the open rows of every segment: a warp each when they are few, else four per warp at a time
  const unsigned found = n_open;  // (the barrier after the last segment ordered it)
  if (flag_total && tid == 0 && found) atomicAdd(flag_total, (unsigned long long)found);
  const int n = (int)min(found, (unsigned)kOpenCap);
  if (n <= 8) {
    if (warp < n)
      decide_grid_warp(set, cbs, n_fixed, s_idx, s_open[warp], out_code, out_ld, out_g0, st, sscale,
                       err);
  }
  for (int e0 = n <= 8 ? n : warp * 4; e0 < n; e0 += 32) {
    const int e = e0 + (lane >> 3);
    decide_grid(set, cbs, n_fixed, s_idx, s_open[min(e, n - 1)], e < n, out_code, out_ld, out_g0,
                st, sscale, err);
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem_slot, 2 * kTcCols);
}

// --------------------------------------------------------------------------- arg-min pass,
// codebooks of more than 256 codewords: a CTA walks `tiles` consecutive row tiles of one group
// (thread = row = tensor-memory lane), streaming the codebook's precomputed B images in chunks of 128
// codewords by bulk copy, in two halves of 128 threads with an accumulator, two chunk buffers, barriers
// and MMA issue each. OWN: a half takes every second tile and all chunks. Otherwise the halves share a
// tile's A rows and take alternate chunks; half 1 hands its minima to half 0 at the tile's end. Two CTAs
// per SM: four pipelines of four warps whose waits (copy, MMA, accumulator loads) overlap. (128 threads
// with two accumulators, so eight warps per SM, took 0.95 us per chunk: one warp per scheduler and CTA
// cannot hide its own load and dependence latency. Shared tiles alone left half 1 idle for the rows,
// certificate and statistics of every tile, most of the work with few chunks: 300 codewords over 12000
// x 512 vectors took 841 us, 596 with a tile per half.)
//
// Sweep, as in argmin_small_kernel but over 32-column granules and 32 classes (column % 32): a
// granule's minimum and the class minima, 0.5 + 0.5 instructions per score, and the three smallest
// granule minima with the first two's numbers (10 instructions per 32 scores). The winner is the
// smallest granule's column of the smallest class; the runner-up is the second smallest granule or
// class minimum. An open row whose third smallest granule lies above the bound has its candidates in
// two granules and the classes below the bound (a few columns): the narrow list (decide_narrow).
// The others (wide list) are decided over the whole codebook. Sending every
// open row over the whole codebook took 60% of a K = 65536 pass (3% of the rows are open there).
struct NarrowRow {
  uint32_t i, g;     // row, group (absolute)
  uint32_t gran;     // the two granules, first << 16 | second (the same twice: one)
  uint32_t classes;  // mask
};

struct NarrowList {
  NarrowRow* row;
  unsigned* count;
  unsigned long long* total;  // optional running total of open rows
};

constexpr int kGran = 32;      // columns per granule
constexpr int kBRing = 2;      // B chunk buffers of a half

constexpr int kHandWords = 5 + kGran;  // half 1's minima of a row
constexpr size_t argmin_stream_smem(bool own) {
  return (own ? 2 : 1) * (size_t)tcenc::kATile + 2 * kBRing * (size_t)kTcBTile +
         (size_t)tcenc::kRows * (own ? 2 * kD : kD + kHandWords) * 4 + 1024;
}

template <bool OWN>
__global__ void __launch_bounds__(256, 2)
argmin_tc_kernel(SetView set, int64_t g_begin, CbList cbs, int n_fixed, int s_idx,
                 int32_t* __restrict__ out_code, int64_t out_ld, int64_t out_g0,
                 FlagList wide, NarrowList narrow, StatsView st, const float* __restrict__ cbmax,
                 const char* __restrict__ bpre, const char* __restrict__ bpre_g, const float4* __restrict__ terms,
                 const float4* __restrict__ rowterms, int tiles, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  using namespace tcenc;
  extern __shared__ __align__(1024) char smem_raw[];
  // 1024-byte aligned base, derived from the shared array (keeps the shared address space)
  char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  const int tid = threadIdx.x, warp = tid >> 5, half = tid >> 7, rrow = tid & (kRows - 1);
  constexpr int kTiles = OWN ? 2 : 1;                     // A tiles at a time
  char* Atile = smem + (OWN ? half : 0) * kATile;         // kTiles x 16 KB
  char* Bbuf = smem + kTiles * kATile + half * kBRing * kTcBTile;  // this half's kBRing x 16 KB
  float* sQ = reinterpret_cast<float*>(smem + kTiles * kATile + 2 * kBRing * kTcBTile) +
              (OWN ? half : 0) * kRows * kD;              // [128][8]: H r
  uint32_t* hand = reinterpret_cast<uint32_t*>(sQ + kRows * kD);  // [kHandWords][128] (not OWN)
  __shared__ __align__(16) float sH[kD * kD];
  __shared__ __align__(8) uint64_t bar_mma_s[2], bar_b_s[2][kBRing];
  __shared__ uint32_t tmem_slot;
  uint64_t& bar_mma = bar_mma_s[half];
  uint64_t* bar_b = bar_b_s[half];

  const int64_t g = g_begin + blockIdx.y;
  const int64_t G_range = gridDim.y;
  const CbView cw = cbs.cb[s_idx];
  const float cmul = kCmul + 4.f * n_fixed;
  const float uc = kU * cmul;
  const int nchunk = (cw.K + kTcCols - 1) / kTcCols;
  const char* bgrp = bpre_g + (size_t)(g - g_begin) * nchunk * kBCol;
  const float4* gterms = terms + (g - g_begin) * cw.K;

  if (tid < kD * kD) sH[tid] = set.Hb[g * kD * kD + tid];
  if (warp == 0) tc::tmem_alloc(&tmem_slot, 2 * kTcCols);
  if (tid == 0) {
    for (int h = 0; h < 2; ++h) {
      tc::mbar_init(tc::smem_u32(&bar_mma_s[h]), 1);
      for (int b = 0; b < kBRing; ++b) tc::mbar_init(tc::smem_u32(&bar_b_s[h][b]), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot + (uint32_t)(half * kTcCols);  // this half's accumulator
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const float sscale = st.cnt ? stats_scale_f(st) : 1.f;

  // Bound on Na_k over the codebook for this group: (max row sum |H_g|) L1max cinfmax.
  float hrow = 0.f;
#pragma unroll
  for (int a = 0; a < kD; ++a) {
    float rs = 0.f;
#pragma unroll
    for (int b = 0; b < kD; ++b) rs += fabsf(sH[a * kD + b]);
    hrow = fmaxf(hrow, rs);
  }
  const float l1max = cbmax[0], cinf = cbmax[1];
  constexpr uint32_t idesc = tc::idesc_tf32(kRows, kTcCols);

  // this CTA's row tiles (the last CTA of a column may have fewer); OWN: half h takes h, h + 2, ...
  const int64_t row_tiles = (set.M + kRows - 1) / kRows;
  const int my_tiles = (int)min((int64_t)tiles, row_tiles - (int64_t)blockIdx.x * tiles);
  const int steps = OWN ? (my_tiles + 1 - half) >> 1 : my_tiles;
  // A half's chunk uses are numbered over its tiles: use u is chunk u % nch of its chunks (all of the
  // codebook's, or every second one), in buffer u % kBRing. The half's thread 0 fetches, waits for and
  // multiplies them in order (fetched: uses whose copy has started, issued: uses whose MMA has).
  const int nch = OWN ? nchunk : (nchunk + 1 - half) >> 1;
  const int64_t n_uses = (int64_t)steps * nch;
  int64_t fetched = 0, issued = 0;
  auto fetch = [&]() {  // the next chunk, into the buffer of the use kBRing before it
    const int b = (int)(fetched % kBRing);
    tc::mbar_expect_tx(tc::smem_u32(&bar_b[b]), kTcBTile);
    const size_t chunk = (size_t)(OWN ? fetched % nch : 2 * (fetched % nch) + half);
    const uint32_t dst = tc::smem_u32(Bbuf + b * kTcBTile), bar = tc::smem_u32(&bar_b[b]);
    const char* src = bpre + chunk * kTcBTile;
    tc::bulk_copy_g2s(dst, src, kBGroupCol * kBCol, bar);
    tc::bulk_copy_g2s(dst + kBGroupCol * kBCol, bgrp + chunk * kBCol, kBCol, bar);
    tc::bulk_copy_g2s(dst + (kBGroupCol + 1) * kBCol, src + (kBGroupCol + 1) * kBCol, kBCol, bar);
    ++fetched;
  };
  // The next use's MMA. After a timeout its waiters are released and the caller's ok turns false.
  auto issue = [&]() -> bool {
    const int b = (int)(issued % kBRing);
    const bool ready = tc::mbar_wait(tc::smem_u32(&bar_b[b]), (uint32_t)((issued / kBRing) & 1), err);
    ++issued;
    if (!ready) {
      tc::mbar_arrive(tc::smem_u32(&bar_mma));
      return false;
    }
    tc::tc_fence_after();
    const uint32_t a0 = tc::smem_u32(Atile), b0 = tc::smem_u32(Bbuf + b * kTcBTile);
#pragma unroll
    for (int ks = 0; ks < kK / 8; ++ks)
      tc::mma_tf32(tmem, tc::smem_desc(a0 + ks * 256, 128, (kK / 4) * 128),
                   tc::smem_desc(b0 + ks * 2 * kBCol, kBCol, 128), idesc, ks > 0 ? 1u : 0u);
    tc::mma_commit(tc::smem_u32(&bar_mma));
    return true;
  };
  if (rrow == 0)
    while (fetched < min((int64_t)kBRing, n_uses)) fetch();
  bool ok = true;
  uint32_t mpar = 0;  // parity of the next MMA wait

  for (int t = 0; t < steps && ok; ++t) {
    const int64_t i = ((int64_t)blockIdx.x * tiles + (OWN ? 2 * t + half : t)) * kRows + rrow;
    const bool row_ok = i < set.M;
    // Prologue: the A rows; of a shared tile by half 0 (which also takes the rows' decisions).
    float pmax = 0.f, off = 0.f;
    if (OWN || half == 0) {
      float m2q[kD], rr, ra;
      if (rowterms) {  // precomputed for this Lloyd loop (row_terms_kernel)
        float4 q0 = make_float4(0.f, 0.f, 0.f, 0.f), q1 = q0, t2 = q0;
        if (row_ok) {
          q0 = rowterms[(3 * g) * set.M + i];
          q1 = rowterms[(3 * g + 1) * set.M + i];
          t2 = rowterms[(3 * g + 2) * set.M + i];
        }
        m2q[0] = q0.x; m2q[1] = q0.y; m2q[2] = q0.z; m2q[3] = q0.w;
        m2q[4] = q1.x; m2q[5] = q1.y; m2q[6] = q1.z; m2q[7] = q1.w;
        rr = t2.x;
        ra = t2.y;
        pmax = t2.z;
      } else {
        float rv[kD], a[kD];
        if (row_ok) {
          target32(set, cbs, n_fixed, i, g, rv, a, err);
        } else {
#pragma unroll
          for (int j = 0; j < kD; ++j) rv[j] = a[j] = 0.f;
        }
        vector_terms_rr(rv, a, sH, m2q, pmax, rr, ra);
      }
      // offset making every D = low + off >= 0, with margins for every rounding involved
      off = (rr + 32.f * kU * ra + 2.f * uc * (hrow * l1max * cinf + 2.f * pmax * l1max)) *
                (1.f + 4.f * uc) + 1e-30f;
      const float beta = -2.f * uc * pmax;
      if (st.cnt) {  // H r of this row, kept for the statistics (-m2q / 2, exact)
        *reinterpret_cast<float4*>(sQ + rrow * kD) =
            make_float4(-0.5f * m2q[0], -0.5f * m2q[1], -0.5f * m2q[2], -0.5f * m2q[3]);
        *reinterpret_cast<float4*>(sQ + rrow * kD + 4) =
            make_float4(-0.5f * m2q[4], -0.5f * m2q[5], -0.5f * m2q[6], -0.5f * m2q[7]);
      }
      uint32_t row[kK];
#pragma unroll
      for (int p = 0; p < kD; ++p) {
        uint32_t h, l;
        split(m2q[p], h, l);
        row[p] = h;
        row[8 + p] = h;
        row[16 + p] = l;
      }
      const uint32_t one = __float_as_uint(1.f);
      row[24] = one;
      row[25] = one;
      split(beta, row[26], row[28]);
      row[27] = row[26];
      split(off * (1.f - uc), row[29], row[30]);
      row[31] = 0u;
      put_row(Atile, rrow, row);
      tc::fence_async_smem();
    }
    if constexpr (OWN)
      half_sync_and(half, true);
    else
      __syncthreads();
    if (rrow == 0) ok = issue();

    // fp32 bits: the three smallest granule minima, the first two's granules; the class minima
    uint32_t v1 = 0xffffffffu, v2 = 0xffffffffu, v3 = 0xffffffffu;
    int b1 = 0, b2 = 0;
    uint32_t mc[kGran];
#pragma unroll
    for (int e = 0; e < kGran; ++e) mc[e] = 0xffffffffu;
    for (int c = 0; c < nch; ++c) {
      const bool done = tc::mbar_wait(tc::smem_u32(&bar_mma), mpar, err);
      mpar ^= 1u;
      ok = __all_sync(0xffffffffu, ok && done);
      tc::tc_fence_after();
      if (ok) {
#pragma unroll
        for (int rnd = 0; rnd < 2; ++rnd) {
          uint32_t v[64];
          tc::tmem_ld64_wait(trow + (uint32_t)(64 * rnd), v);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const uint32_t m = min(min16_bits(v + kGran * q), min16_bits(v + kGran * q + 16));
            const int gr = (OWN ? c : 2 * c + half) * (kTcCols / kGran) + 2 * rnd + q;
            const bool lt1 = m < v1, lt2 = m < v2;
            v3 = min(v3, max(v2, m));
            b2 = lt1 ? b1 : (lt2 ? gr : b2);
            b1 = lt1 ? gr : b1;
            v2 = min(v2, max(v1, m));
            v1 = min(v1, m);
          }
#pragma unroll
          for (int e = 0; e < kGran; ++e) mc[e] = __vimin3_u32(mc[e], v[e], v[kGran + e]);
        }
      }
      tc::tc_fence_before();
      // the accumulator has been read and its MMA is done with its buffer
      ok = half_sync_and(half, ok);
      if (!ok) break;
      if (rrow == 0) {
        if (fetched < n_uses) fetch();
        if (c + 1 < nch) ok = issue();
      }
    }
    if constexpr (OWN) {
      if (!ok) break;
    } else {
      if (half == 1 && ok) {
        hand[0 * kRows + rrow] = v1;
        hand[1 * kRows + rrow] = v2;
        hand[2 * kRows + rrow] = v3;
        hand[3 * kRows + rrow] = (uint32_t)b1;
        hand[4 * kRows + rrow] = (uint32_t)b2;
#pragma unroll
        for (int e = 0; e < kGran; ++e) hand[(5 + e) * kRows + rrow] = mc[e];
      }
      ok = __syncthreads_and(ok);
      if (!ok) break;
      if (half == 1) continue;  // (the next barrier is the next tile's, after its A rows)
      // half 1's granules and classes
      const uint32_t hv[3] = {hand[rrow], hand[kRows + rrow], hand[2 * kRows + rrow]};
      const int hb[3] = {(int)hand[3 * kRows + rrow], (int)hand[4 * kRows + rrow], 0};
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const uint32_t m = hv[q];
        const bool lt1 = m < v1, lt2 = m < v2;
        v3 = min(v3, max(v2, m));
        b2 = lt1 ? b1 : (lt2 ? hb[q] : b2);
        b1 = lt1 ? hb[q] : b1;
        v2 = min(v2, max(v1, m));
        v1 = min(v1, m);
      }
#pragma unroll
      for (int e = 0; e < kGran; ++e) mc[e] = min(mc[e], hand[(5 + e) * kRows + rrow]);
    }

    // Certificate, code, open row and statistics of this thread's row.
    if (row_ok) {
      uint32_t x1, x2;
      int e1;
      top2<kGran>(mc, x1, x2, e1);
      int j = b1 * kGran + e1;
      const uint32_t s2 = min(v2, x2);
      const float k1 = __uint_as_float(v1);
      const float k2 = s2 == 0xffffffffu ? INFINITY : __uint_as_float(s2);
      bool cert = false;
      float thr = INFINITY, top = INFINITY;
      if (j < cw.K) {
        const float4 tj = gterms[j];
        const float na = tj.y, l1 = tj.z;
        // D_k <= s_k + off (every k); s_j + off <= D_j + e2 (the winner): no other codeword's
        // exact score reaches s_j when k2 > D_j + e2 (the sum rounded up).
        float e2 = 2.f * uc * (na + 2.f * pmax * l1 + off);
        top = __fadd_ru(k1, e2);   // >= s_j + off
        cert = k2 > top;
        if (s2 == v1) {
          // Equal scores: granule and class may name different columns. Granule b1 holds a smallest
          // score, in one of the classes that have it: the largest bound among those. (With the bound
          // over the whole codebook such rows were open over most of it: 34.4 instead of 25.2 ms for
          // K = 65536, 1024 x 11008.)
          for (uint32_t em = mask_le<kGran>(mc, v1); em; em &= em - 1u) {
            const int k = b1 * kGran + __ffs(em) - 1;
            if (k >= cw.K) continue;
            const float4 tk = gterms[k];
            e2 = fmaxf(e2, 2.f * uc * (tk.y + 2.f * pmax * tk.z + off));
          }
          top = __fadd_ru(k1, e2);
        }
        thr = top - off;
        thr += 4.f * kU * (k1 + off + e2);
      } else {
        j = 0;
      }
      if (!cert) {
        const uint32_t tb = __float_as_uint(top) & 0x7fffffffu;
        if (v3 > tb && v1 <= tb) {
          const unsigned slot = atomicAdd(narrow.count, 1u);  // at most one per row: it fits
          narrow.row[slot] = NarrowRow{(uint32_t)i, (uint32_t)g,
                                       (uint32_t)b1 << 16 | (uint32_t)(v2 <= tb ? b2 : b1),
                                       mask_le<kGran>(mc, tb)};
        } else {
          const unsigned slot = atomicAdd(wide.count, 1u);
          if (slot < wide.cap) {
            wide.vec[slot] = i * G_range + (g - g_begin);
            wide.thr[slot] = thr;
          } else {
            raise_error(err, ERRBIT_INDEX);
          }
        }
      }
      if (out_code) out_code[i * out_ld + (g - out_g0)] = j;
      if (cert && st.cnt) {
        // H r from the prologue (bit-identical to the standalone update's H tau)
        float q[kD];
        const float4 q0 = *reinterpret_cast<const float4*>(sQ + rrow * kD);
        const float4 q1 = *reinterpret_cast<const float4*>(sQ + rrow * kD + 4);
        q[0] = q0.x; q[1] = q0.y; q[2] = q0.z; q[3] = q0.w;
        q[4] = q1.x; q[5] = q1.y; q[6] = q1.z; q[7] = q1.w;
        stats_add(st, sscale, g, j, q);
      }
    }
  }
  // After a timeout: let copies still in flight into this CTA's shared memory land (bounded).
  if (rrow == 0)
    for (; issued < fetched; ++issued)
      tc::mbar_wait(tc::smem_u32(&bar_b[issued % kBRing]), (uint32_t)((issued / kBRing) & 1), err);
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem_slot, 2 * kTcCols);
}

// Exact decision of the narrow list, a quarter warp per row, by every warp of the grid.
__device__ __forceinline__ void decide_narrow(const SetView& set, const CbList& cbs, int n_fixed,
                                              int s_idx, int32_t* __restrict__ out_code,
                                              int64_t out_ld, int64_t out_g0, const NarrowList& list,
                                              const StatsView& st, unsigned* err) {
  const int n = (int)*list.count;
  if (list.total && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(list.total, (unsigned long long)n);
  const float sscale = st.cnt ? stats_scale_f(st) : 1.f;
  const int quarter = (threadIdx.x & 31) >> 3;
  const int warps = (int)(blockDim.x >> 5);
  for (int e0 = (blockIdx.x * warps + (threadIdx.x >> 5)) * 4; e0 < n; e0 += gridDim.x * warps * 4) {
    const int e = e0 + quarter;
    const NarrowRow o = list.row[min(e, n - 1)];
    const int ga = (int)(o.gran >> 16), gb = (int)(o.gran & 0xffffu), ne = __popc(o.classes);
    decide_open(set, cbs, n_fixed, s_idx, o.i, o.g, e < n, (ga == gb ? 1 : 2) * ne,
                [&](int c) { return kGran * (c < ne ? ga : gb) + nth_bit(o.classes, c % ne); },
                out_code, out_ld, out_g0, st, sscale, err);
  }
}

// Whether c equals codeword k (an index past the codebook: no). A thread's candidate that repeats its best so
// far cannot win, and is not scored (see argmin_small_kernel on repeated codewords).
__device__ __forceinline__ bool equals(const CbView& cw, int k, const float c[kD]) {
  if (k >= cw.K) return false;
  float o[kD];
  load_vec(cw.C + (int64_t)k * kD, o);
  bool same = true;
#pragma unroll
  for (int j = 0; j < kD; ++j) same = same && c[j] == o[j];
  return same;
}

// Exact decision of rows open over the whole codebook (argmin_tc_kernel's wide list): one CTA per row.
// The threads stride over the codebook for U = min(fast-pass threshold, smallest fp32 upper
// bound); every codeword whose fp32 lower bound is at most U is a candidate (the exact
// arg-min always is) and is re-scored exactly in fp32 pairs (dfl) by the thread that holds it; the
// smallest (err, index) wins. Adds the statistics of the decided code when requested. A launch with a
// single such row takes as long as its scan: kExactThreads threads with kWideBatch codewords in
// flight each (128 threads with one took 0.75 ms for 65536 codewords).
constexpr int kExactThreads = 512;
constexpr int kWideBatch = 4;  // codewords a thread loads before using them

__global__ void __launch_bounds__(kExactThreads)
argmin_exact_kernel(SetView set, int64_t g_begin, int64_t G_range, CbList cbs, int n_fixed,
                    int s_idx, int32_t* __restrict__ out_code, int64_t out_ld, int64_t out_g0,
                    FlagList flags, unsigned many, StatsView st,
                    const float4* __restrict__ terms, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  constexpr int kWarps = kExactThreads / 32;
  __shared__ float sH[kD * kD];
  __shared__ float redf[kWarps];
  __shared__ float bh_s[kWarps], bl_s[kWarps];
  __shared__ int bk_s[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned cnt = min((unsigned long long)*flags.count, (unsigned long long)flags.cap);
  if (cnt > many) return;  // (argmin_exact_warp_kernel has taken them)
  if (flags.total && blockIdx.x == 0 && tid == 0) atomicAdd(flags.total, cnt);
  const CbView cw = cbs.cb[s_idx];
  const float cmul = bound_mult(n_fixed);
  for (unsigned f = blockIdx.x; f < cnt; f += gridDim.x) {
    const int64_t vi = flags.vec[f];
    const int64_t i = vi / G_range, grel = vi % G_range, g = g_begin + grel;
    __syncthreads();
    if (tid < kD * kD) sH[tid] = set.Hb[g * kD * kD + tid];
    __syncthreads();
    float rv[kD], av[kD], m2q[kD], pmax;
    target32(set, cbs, n_fixed, i, g, rv, av, err);
    vector_terms(rv, av, sH, m2q, pmax);
    const float nbeta = -2.f * kU * cmul * pmax;
    const float4* gt = terms + grel * cw.K;
    // two passes over the codebook: f(k, codeword, n, Na, L1)
    auto sweep = [&](auto f) {
      for (int k0 = tid; k0 < cw.K; k0 += kExactThreads * kWideBatch) {
        float cv[kWideBatch][kD];
        float4 tt[kWideBatch];
#pragma unroll
        for (int u = 0; u < kWideBatch; ++u) {
          const int k = min(k0 + u * kExactThreads, cw.K - 1);  // (the last one again past the end)
          load_vec(cw.C + (int64_t)k * kD, cv[u]);
          tt[u] = gt[k];
        }
#pragma unroll
        for (int u = 0; u < kWideBatch; ++u)
          f(min(k0 + u * kExactThreads, cw.K - 1), cv[u], tt[u].x, tt[u].y, tt[u].z);
      }
    };
    float U = flags.thr[f];
    sweep([&](int, const float cv[kD], float nn, float na, float l1) {
      U = fminf(U, up_from(nn, na, l1, cv, m2q, pmax, cmul));
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) U = fminf(U, __shfl_xor_sync(0xffffffffu, U, o));
    if (lane == 0) redf[warp] = U;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kWarps; ++w) U = fminf(U, redf[w]);
    float rh[kD], rl[kD];
    dfl::target(set, cbs, n_fixed, i, g, rh, rl, err);
    float bh = INFINITY, bl = 0.f;
    int bk = 0x7fffffff;
    sweep([&](int k, const float cv[kD], float nn, float na, float l1) {
      if (low_from(nn, na, l1, cv, m2q, nbeta, cmul) <= U && !equals(cw, bk, cv)) {
        float eh, el;
        dfl::quad_err(rh, rl, cv, sH, eh, el);
        if (dfl::less(eh, el, k, bh, bl, bk)) {
          bh = eh;
          bl = el;
          bk = k;
        }
      }
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, bh, o);
      const float ol = __shfl_xor_sync(0xffffffffu, bl, o);
      const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
      if (dfl::less(oh, ol, ok, bh, bl, bk)) {
        bh = oh;
        bl = ol;
        bk = ok;
      }
    }
    if (lane == 0) {
      bh_s[warp] = bh;
      bl_s[warp] = bl;
      bk_s[warp] = bk;
    }
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < kWarps; ++w)
        if (dfl::less(bh_s[w], bl_s[w], bk_s[w], bh, bl, bk)) {
          bh = bh_s[w];
          bl = bl_s[w];
          bk = bk_s[w];
        }
      if (bk == 0x7fffffff) {
        raise_error(err, ERRBIT_NUMERIC);  // no candidate: non-finite scores
      } else {
        if (out_code) out_code[i * out_ld + (g - out_g0)] = bk;
        if (st.cnt) {
          float q[kD];
#pragma unroll
          for (int p = 0; p < kD; ++p) q[p] = -0.5f * m2q[p];
          stats_add(st, stats_scale_f(st), g, bk, q);
        }
      }
    }
  }
}


// Exact decision of both open lists: the narrow one, then the wide one with a warp per row, by the bounds
// and fp32-pair scores of argmin_exact_kernel without block barriers. Lane l takes codewords l, l + 32,
// ...; the fp32 upper bounds give U, every codeword whose lower bound reaches U is scored in fp32 pairs
// by the lane that holds it, and the best (value, index) is reduced across the warp with the same total
// order, so the decision is the one argmin_exact_kernel makes. Wide lists of at most `many` rows are left
// to that kernel: above kExactWarpK codewords a lone row is a long scan for a warp, but with thousands of
// them (a matrix full of repeated vectors) a block each wastes its barriers and most of its threads
// (4096 codewords, half of 1024 x 512 vectors open: 38 ms by blocks, 14 by warps).
constexpr int kExactWarpK = 1024;
constexpr int kExactBatch = 2;  // codewords a lane loads before using them

__global__ void __launch_bounds__(128)
argmin_exact_warp_kernel(SetView set, int64_t g_begin, int64_t G_range, CbList cbs,
                         int n_fixed, int s_idx, int32_t* __restrict__ out_code, int64_t out_ld,
                         int64_t out_g0, NarrowList narrow, FlagList flags, unsigned many, StatsView st,
                         const float4* __restrict__ terms, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  decide_narrow(set, cbs, n_fixed, s_idx, out_code, out_ld, out_g0, narrow, st, err);
  __shared__ float sHw[4][kD * kD];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned cnt = min((unsigned long long)*flags.count, (unsigned long long)flags.cap);
  if (cnt <= many) return;  // (left to argmin_exact_kernel)
  if (flags.total && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(flags.total, cnt);
  const CbView cw = cbs.cb[s_idx];
  const float cmul = bound_mult(n_fixed);
  float* sH = sHw[warp];
  for (unsigned f = blockIdx.x * 4u + warp; f < cnt; f += gridDim.x * 4u) {
    const int64_t vi = flags.vec[f];
    const int64_t i = vi / G_range, grel = vi % G_range, g = g_begin + grel;
    const float thr = flags.thr[f];
    __syncwarp();
    sH[lane] = set.Hb[g * kD * kD + lane];
    sH[lane + 32] = set.Hb[g * kD * kD + lane + 32];
    __syncwarp();
    float rv[kD], av[kD], m2q[kD], pmax;
    target32(set, cbs, n_fixed, i, g, rv, av, err);
    vector_terms(rv, av, sH, m2q, pmax);
    const float nbeta = -2.f * kU * cmul * pmax;
    const float4* gt = terms + grel * cw.K;
    // a lane takes codewords lane, lane + 32, ...; kExactBatch of them are loaded before any is
    // used, so their L2 round trips overlap
    float U = thr;
    for (int k0 = lane; k0 < cw.K; k0 += 32 * kExactBatch) {
      float cv[kExactBatch][kD];
      float4 tt[kExactBatch];
#pragma unroll
      for (int u = 0; u < kExactBatch; ++u) {
        const int k = k0 + 32 * u;
        if (k < cw.K) {
          load_vec(cw.C + (int64_t)k * kD, cv[u]);
          tt[u] = gt[k];
        }
      }
#pragma unroll
      for (int u = 0; u < kExactBatch; ++u) {
        if (k0 + 32 * u >= cw.K) break;
        U = fminf(U, up_from(tt[u].x, tt[u].y, tt[u].z, cv[u], m2q, pmax, cmul));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) U = fminf(U, __shfl_xor_sync(0xffffffffu, U, o));
    float rh[kD], rl[kD];
    dfl::target(set, cbs, n_fixed, i, g, rh, rl, err);
    float bh = INFINITY, bl = 0.f;
    int bk = 0x7fffffff;
    for (int k = lane; k < cw.K; k += 32) {
      float cv[kD];
      load_vec(cw.C + (int64_t)k * kD, cv);
      const float4 t = gt[k];
      if (low_from(t.x, t.y, t.z, cv, m2q, nbeta, cmul) <= U && !equals(cw, bk, cv)) {
        float eh, el;
        dfl::quad_err(rh, rl, cv, sH, eh, el);
        if (dfl::less(eh, el, k, bh, bl, bk)) {
          bh = eh;
          bl = el;
          bk = k;
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, bh, o);
      const float ol = __shfl_xor_sync(0xffffffffu, bl, o);
      const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
      if (dfl::less(oh, ol, ok, bh, bl, bk)) {
        bh = oh;
        bl = ol;
        bk = ok;
      }
    }
    if (lane == 0) {
      if (bk == 0x7fffffff) {
        raise_error(err, ERRBIT_NUMERIC);  // no candidate: non-finite scores
      } else {
        if (out_code) out_code[i * out_ld + (g - out_g0)] = bk;
        if (st.cnt) {
          float q[kD];
#pragma unroll
          for (int p = 0; p < kD; ++p) q[p] = -0.5f * m2q[p];
          stats_add(st, stats_scale_f(st), g, bk, q);
        }
      }
    }
  }
}

// --------------------------------------------------------------------------- beam stages
// Hypotheses of a vector: up to B partial tuples (codes of the first s+1 searched codebooks)
// in rank order. hyp layout: [vector][B][S] int32; hyp_n[vector] = number kept.
struct BeamBufs {
  const int32_t* hyp_in;
  const int32_t* n_in;
  int32_t* hyp_out;
  int32_t* n_out;
};

struct StageDesc {
  int st[kMaxCodebooks];  // indices (in cbs) of the searched codebooks, in stage order
  int S;                  // number of stages
  int s;                  // current stage
  int B;                  // beam width (hypothesis buffer stride)
  int Bs;                 // hypotheses kept by the current stage (1 at the last stage)
};

// fp32-pair residual of a hypothesis before stage s: (rh + rl) = (th + tl) - sum_{s' < s}
// C_{st[s']}[code] (TwoSum per subtraction, about 2^-48 relative; no fp64 arithmetic).
__device__ __forceinline__ void hyp_residual_pair(const float th[kD], const float tl[kD],
                                                  const CbList& cbs, const StageDesc& sd,
                                                  const int32_t* codes, float rh[kD],
                                                  float rl[kD], unsigned* err) {
#pragma unroll
  for (int j = 0; j < kD; ++j) {
    rh[j] = th[j];
    rl[j] = tl[j];
  }
  for (int q = 0; q < sd.s; ++q) {
    const CbView& cb = cbs.cb[sd.st[q]];
    const int32_t k = codes[q];
    if (!code_ok(k, cb.K, err)) continue;
    float c[kD];
    load_vec(cb.C + (int64_t)k * kD, c);
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      float sj, ej;
      dfl::two_sum(rh[j], -c[j], sj, ej);
      rh[j] = sj;
      rl[j] = __fadd_rn(rl[j], ej);
    }
  }
}

// Per-hypothesis terms of the approximate err: m2q = -2 H r, rr = r^T H r (r: the pair residual
// rounded to fp32), and the bound pieces Ra = |r|^T |H| |r|, Pmax = max_p (|H| |r|)_p.
__device__ __forceinline__ void hyp_terms_pair(const float rh[kD], const float rl[kD],
                                               const float* H, float m2q[kD], float& rr,
                                               float& ra, float& pmax) {
  float r[kD];
#pragma unroll
  for (int j = 0; j < kD; ++j) r[j] = __fadd_rn(rh[j], rl[j]);
  rr = 0.f;
  ra = 0.f;
  pmax = 0.f;
#pragma unroll
  for (int p = 0; p < kD; ++p) {
    float q = 0.f, pa = 0.f;
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      q = fmaf(H[p * kD + j], r[j], q);
      pa = fmaf(fabsf(H[p * kD + j]), fabsf(r[j]), pa);
    }
    m2q[p] = -2.f * q;
    rr = fmaf(r[p], q, rr);
    ra = fmaf(fabsf(r[p]), pa, ra);
    pmax = fmaxf(pmax, pa);
  }
}

// The end of a fast stage, given each thread's sorted top-L list (topv, topi) of fp32 lower bounds
// low = approx_err - Et built in (h, k) order: bounds of the listed entries, the fast certificate,
// the exact decision in fp32 pairs, the flag for the fallback, and the kept tuples. Whole warps call
// it; a thread with live = false has no vector and only helps.
// sRa / sPm: Ra_h, Pmax_h of this thread's hypotheses at [h * stride]; sNL / sNa: the staged
// codeword terms (used when the whole codebook was staged, else recomputed).
//
// Exact decisions: a few vectors per warp fail the fast certificate, and their L entries cost about
// 700 instructions each, so a lane takes one entry: 32 / L vectors at a time, ranks among a
// vector's entries by shuffles, the entry of rank r writes tuple r. (A thread deciding all entries of
// its own vector kept the warp for L entries whenever one lane had to: three stages over 11008 x 11
// vectors with 8 hypotheses took 874 us, now 655.)
template <int L>
__device__ __forceinline__ void beam_list_finish(
    const SetView& set, const CbList& cbs, const StageDesc& sd, const BeamBufs& bb,
    const FlagList& flags, bool live, int64_t i, int64_t g, int64_t vi, int Bh, float cmul,
    const float th[kD], const float tl[kD], const float* sH, const float2* sNL,
    const float* sNa, bool one_chunk, const float* sRa, const float* sPm, int stride,
    float topv[L], int topi[L], unsigned* err) {
  const CbView cw = cbs.cb[sd.st[sd.s]];
  const int S = sd.S, B = sd.B, Bs = sd.Bs;
  const int lane = threadIdx.x & 31;
  bool open = false;
  if (live) {
    const int64_t total = (int64_t)Bh * cw.K;
    const int nkept = (int)min((int64_t)L, total);
    const int keep = (int)min((int64_t)Bs, total);
    // Non-finite scores never enter the list; keep indices valid and report it.
#pragma unroll
    for (int j = 0; j < L; ++j) {
      if (j < nkept && ((topi[j] >> 16) >= Bh || (topi[j] & 0xffff) >= cw.K)) {
        raise_error(err, ERRBIT_NUMERIC);
        topi[j] = 0;
      }
    }
    // Fast certificate: low_{j+1} - low_j > 2 Et_j for j < min(keep, total - 1) (every candidate
    // outside the list has low >= the last list entry), with the per-entry bound
    // Et = u C (Ra_h + Na_k + 2 Pmax_h L1_k) from the hypothesis terms kept in the sweep and the
    // staged codeword terms (recomputed when the codebook spans several chunks).
    const int lim = (int)min((int64_t)keep, total - 1);
#pragma unroll
    for (int j = 0; j < L - 1; ++j) {
      if (j < lim) {
        const int h = topi[j] >> 16, k = topi[j] & 0xffff;
        float na, l1;
        if (one_chunk) {
          na = sNa[k];
          l1 = sNL[k].y;
        } else {
          float c[kD], n;
          load_vec(cw.C + (int64_t)k * kD, c);
          codeword_terms(c, sH, n, na, l1);
        }
        const float et = kU * cmul * (sRa[h * stride] + na + 2.f * sPm[h * stride] * l1);
        if (!(topv[j + 1] - topv[j] > 2.f * et)) open = true;
      }
    }
    if (!open) {
      int32_t* out = bb.hyp_out + vi * B * S;
#pragma unroll
      for (int j = 0; j < L; ++j) {
        if (j >= keep) break;
        const int32_t* pc = bb.hyp_in ? bb.hyp_in + (vi * B + (topi[j] >> 16)) * S : nullptr;
        for (int q = 0; q < sd.s; ++q) out[j * S + q] = pc[q];
        out[j * S + sd.s] = topi[j] & 0xffff;
      }
      bb.n_out[vi] = keep;
    }
  }
  // Exact decisions: lane = (slot, entry) of the next 32 / L open vectors. Errs as fp32 pairs (about
  // 2^-44 of their terms; no fp64) in (err, h, k) order; every unlisted candidate must have low >= the
  // last listed low, which must exceed an upper bound of the keep-th err.
  constexpr int kPer = 32 / L;
  const int slot = lane / L, e = lane - slot * L;
  unsigned todo = __ballot_sync(0xffffffffu, open);
  while (todo) {
    unsigned rest = todo;
    int src = -1;
    for (int q = 0; q < kPer && rest; ++q) {
      if (q == slot) src = __ffs(rest) - 1;
      rest &= rest - 1u;
    }
    const bool has = src >= 0;
    const int from = has ? src : __ffs(todo) - 1;
    todo = rest;
    float vth[kD], vtl[kD];
#pragma unroll
    for (int q = 0; q < kD; ++q) {
      vth[q] = __shfl_sync(0xffffffffu, th[q], from);
      vtl[q] = __shfl_sync(0xffffffffu, tl[q], from);
    }
    const int64_t v = __shfl_sync(0xffffffffu, vi, from);
    const int64_t total = (int64_t)__shfl_sync(0xffffffffu, Bh, from) * cw.K;
    const int nkept = (int)min((int64_t)L, total);
    const int keep = (int)min((int64_t)Bs, total);
    int hk = 0;
    float last_low = INFINITY;
#pragma unroll
    for (int j = 0; j < L; ++j) {
      const int t = __shfl_sync(0xffffffffu, topi[j], from);
      const float x = __shfl_sync(0xffffffffu, topv[j], from);
      if (j == e) hk = t;
      if (j == nkept - 1) last_low = x;
    }
    const bool mine = has && e < nkept;
    float eh = INFINITY, el = 0.f;
    const int32_t* pc = bb.hyp_in ? bb.hyp_in + (v * B + (hk >> 16)) * S : nullptr;
    if (mine) {
      float rh[kD], rl[kD], c[kD];
      hyp_residual_pair(vth, vtl, cbs, sd, pc, rh, rl, err);
      load_vec(cw.C + (int64_t)(hk & 0xffff) * kD, c);
      dfl::quad_err(rh, rl, c, sH, eh, el);
      if (!isfinite(eh)) {  // (NaN too: the ranks stay a permutation)
        eh = INFINITY;
        el = 0.f;
      }
    }
    __syncwarp();
    // rank among the vector's entries by (err, (h, k)), then place
    int rank = 0;
#pragma unroll
    for (int j = 0; j < L; ++j) {
      const int at = min(slot * L + j, 31);
      const float oh = __shfl_sync(0xffffffffu, eh, at), ol = __shfl_sync(0xffffffffu, el, at);
      const int ok = __shfl_sync(0xffffffffu, hk, at);
      const bool same = oh == eh && ol == el && ok == hk;
      if (j < nkept && (same ? j < e : dfl::less(oh, ol, ok, eh, el, hk))) ++rank;
    }
    const unsigned holder =
        (__ballot_sync(0xffffffffu, mine && rank == keep - 1) >> min(slot * L, 31)) &
        ((1u << L) - 1u);
    const int kth = holder ? min(slot * L + __ffs(holder) - 1, 31) : lane;
    const float kh = __shfl_sync(0xffffffffu, eh, kth), kl = __shfl_sync(0xffffffffu, el, kth);
    // upper bound of the keep-th listed err (the pair's own error is far below 1e-7)
    const float ev_up = isfinite(kh) ? __fmul_ru(__fadd_ru(kh, kl), 1.0000002f) : INFINITY;
    const bool cert = total <= L || last_low > ev_up;
    if (mine && cert && rank < keep) {
      int32_t* out = bb.hyp_out + (v * B + rank) * S;
      for (int q = 0; q < sd.s; ++q) out[q] = pc[q];
      out[sd.s] = hk & 0xffff;
    }
    if (has && e == 0) {
      if (cert) {
        bb.n_out[v] = keep;
      } else {
        const unsigned at = atomicAdd(flags.count, 1u);
        if (at < flags.cap) {
          flags.vec[at] = v;
          // every member of the exact top-keep has err <= the keep-th listed err
          flags.thr[at] = ev_up;
        } else {
          raise_error(err, ERRBIT_INDEX);
        }
      }
    }
  }
}

constexpr int kBeamCand = 16;  // candidate buffer slots per thread
constexpr int kBeamScan = 8;   // scores between two overflow checks

// Fast stage: one thread per vector, the stage codebook chunked through shared memory, a
// sorted top-L list (L >= Bs + 1) of lower bounds low = approx_err - Et in registers.
template <int L>
__global__ void __launch_bounds__(kThreads, L <= 9 ? 3 : 2)
beam_stage_kernel(SetView set, int64_t g_begin, CbList cbs, int n_fixed, StageDesc sd,
                  BeamBufs bb, FlagList flags, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const int64_t g = g_begin + blockIdx.y;
  const int64_t G_range = gridDim.y;
  const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const bool live = i < set.M;
  const int64_t vi = live ? i * G_range + (g - g_begin) : 0;
  __shared__ float sH[kD * kD];
  __shared__ __align__(16) float sC[kChunk * kD];
  __shared__ __align__(8) float2 sNL[kChunk];
  __shared__ float sNa[kChunk];
  // candidate buffers, [slot][thread]: (score bits, (h << 16) | k)
  __shared__ uint2 cand[kBeamCand * kThreads];
  __shared__ float sRa[16 * kThreads], sPm[16 * kThreads];  // Ra_h, Pmax_h, [h][thread]
  if (threadIdx.x < kD * kD) sH[threadIdx.x] = set.Hb[g * kD * kD + threadIdx.x];
  __syncthreads();

  const CbView cw = cbs.cb[sd.st[sd.s]];
  const int S = sd.S, B = sd.B;
  const float cmul = bound_mult(n_fixed + sd.s);
  const int Bh = (sd.s == 0) ? 1 : (live ? bb.n_in[vi] : 1);
  float th[kD], tl[kD];  // target as an fp32 pair (t - the fixed codebooks' codewords)
  if (live) {
    dfl::target(set, cbs, n_fixed, i, g, th, tl, err);
  } else {
#pragma unroll
    for (int j = 0; j < kD; ++j) th[j] = tl[j] = 0.f;
  }

  float topv[L];
  int topi[L];  // (h << 16) | k: B <= 16 hypotheses, K <= 65536 codewords
#pragma unroll
  for (int j = 0; j < L; ++j) {
    topv[j] = INFINITY;
    topi[j] = 0x7fffffff;
  }

  // Scores below the list's last entry (as of the last flush) are appended to this thread's
  // candidate buffer in shared memory: a predicated store per score, no branch. Every kBeamScan
  // scores the warp flushes when any lane's buffer could overflow within the next stretch:
  // the buffered candidates, in (h, k) order, go through the sorted insertion (ties keep the
  // earlier candidate ahead, as inserting every score in order would). The insertion network,
  // which the compiler predicates, thus runs per candidate instead of per score.
  int nc = 0;
  float thr = INFINITY;
  auto flush = [&]() {
    for (int e = 0; e < nc; ++e) {
      const uint2 ce = cand[e * kThreads + threadIdx.x];
      float sv = __uint_as_float(ce.x);
      int si = (int)ce.y;
      if (sv < topv[L - 1]) {
#pragma unroll
        for (int j = 0; j < L; ++j) {
          if (sv < topv[j]) {
            const float tv = topv[j];
            const int ti = topi[j];
            topv[j] = sv;
            topi[j] = si;
            sv = tv;
            si = ti;
          }
        }
      }
    }
    nc = 0;
    thr = topv[L - 1];
  };
  for (int k0 = 0; k0 < cw.K; k0 += kChunk) {
    const int nk = min(kChunk, cw.K - k0);
    __syncthreads();
    stage_chunk(cw.C, k0, nk, sH, cmul, sC, sNL, sNa);
    __syncthreads();
    if (!live) continue;
    for (int h = 0; h < Bh; ++h) {
      float rh[kD], rl[kD];
      const int32_t* pc = bb.hyp_in ? bb.hyp_in + (vi * B + h) * S : nullptr;
      hyp_residual_pair(th, tl, cbs, sd, pc, rh, rl, err);
      float m2q[kD], rr, ra, pmax;
      hyp_terms_pair(rh, rl, sH, m2q, rr, ra, pmax);
      sRa[h * kThreads + threadIdx.x] = ra;  // the same values in every chunk
      sPm[h * kThreads + threadIdx.x] = pmax;
      const float base = rr - kU * cmul * ra;
      const float nbeta = -2.f * kU * cmul * pmax;
      // One score: a chain of ten dependent operations; four independent chains per step.
      // Every score is stored into slot nc, which advances only for a candidate (no branch);
      // nc <= kBeamCand - kBeamScan after each check, so the at most kBeamScan stores that
      // follow stay below kBeamCand.
      auto score_at = [&](int k) {
        const float4 c0 = *reinterpret_cast<const float4*>(sC + k * kD);
        const float4 c1 = *reinterpret_cast<const float4*>(sC + k * kD + 4);
        const float2 nl = sNL[k];
        float sc = base + nl.x;
        sc = fmaf(m2q[0], c0.x, sc);
        sc = fmaf(m2q[1], c0.y, sc);
        sc = fmaf(m2q[2], c0.z, sc);
        sc = fmaf(m2q[3], c0.w, sc);
        sc = fmaf(m2q[4], c1.x, sc);
        sc = fmaf(m2q[5], c1.y, sc);
        sc = fmaf(m2q[6], c1.z, sc);
        sc = fmaf(m2q[7], c1.w, sc);
        return fmaf(nbeta, nl.y, sc);
      };
      const uint32_t hk = ((uint32_t)h << 16) | (uint32_t)k0;
      for (int kb = 0; kb < nk; kb += kBeamScan) {
        if (__any_sync(__activemask(), nc > kBeamCand - kBeamScan)) flush();
        if (kb + kBeamScan <= nk) {
#pragma unroll
          for (int e0 = 0; e0 < kBeamScan; e0 += 4) {
            float sc[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) sc[e] = score_at(kb + e0 + e);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              cand[nc * kThreads + threadIdx.x] =
                  make_uint2(__float_as_uint(sc[e]), hk + (uint32_t)(kb + e0 + e));
              nc += sc[e] < thr ? 1 : 0;
            }
          }
        } else {
          for (int k = kb; k < nk; ++k) {
            const float s1 = score_at(k);
            cand[nc * kThreads + threadIdx.x] =
                make_uint2(__float_as_uint(s1), hk + (uint32_t)k);
            nc += s1 < thr ? 1 : 0;
          }
        }
      }
    }
  }
  if (live) flush();
  __syncwarp();
  beam_list_finish<L>(set, cbs, sd, bb, flags, live, i, g, vi, Bh, cmul, th, tl, sH, sNL, sNa,
                      cw.K <= kChunk, sRa + threadIdx.x, sPm + threadIdx.x, kThreads, topv,
                      topi, err);
}

// Fast stage with the scores on the tensor cores (codebooks of at most 256 codewords, L <= 9).
// Thread = vector, as in beam_stage_kernel; the CTA's 128 vectors take the hypotheses in turn:
// for hypothesis h every thread writes its A row, one tcgen05.mma pass computes
//   y(h, k) = base_h + sN_k + m2q_h . c_k + nbeta_h L1_k
// for all 128 vectors x 256 codewords (3xTF32 operands: the B images of prep_b built with the
// stage's bound multiplier), and each thread reads its row from tensor memory. y differs from
// the fast stage's fp32 chain x(h, k) (the same linear form) by at most eps_h = 2^-16 S_h,
// S_h = |base_h| + Na_max + 2 Pmax_h L1max + |nbeta_h| L1max, which bounds every term's
// magnitude (the split products lose about 2^-22 and the fp32 accumulation of 32 terms about
// 2^-19 of it; the arg-min pass's bound multiplier of 256 u is the same 2^-16). Outlier codewords
// make S_h large against the errs, so a looser eps lets many pairs through: at 2^-12 candidates
// were most of the kernel's instructions. A pair whose x could enter the list has y <= (the list's last x, or the bound
// tau below) + eps_h; only those are kept (a bit mask per thread), scored again with exactly
// the fast stage's chain and inserted in (h, k) order with its rule (strictly below the last
// entry, before the first entry strictly above). Every member of the final
// top-L is among them, so the list, and everything after it (beam_list_finish), equals
// beam_stage_kernel's. tau: for h = 0, the L-th smallest of the 16-column block minima of y:
// at least L pairs have y <= tau, so the L-th smallest x is at most tau + eps_0.
constexpr size_t kBeamTcSmem = 1024 + (size_t)tcenc::kATile + 2 * (size_t)kTcBTile +
                               (size_t)kChunk * kD * 4 + (size_t)kChunk * 8 + (size_t)kChunk * 4 +
                               2 * 16 * (size_t)kThreads * 4 + 8 * (size_t)kThreads * 4;

template <int L>
__global__ void __launch_bounds__(kThreads, 2)
beam_tc_kernel(SetView set, int64_t g_begin, CbList cbs, int n_fixed, StageDesc sd,
               BeamBufs bb, const char* __restrict__ bimg, const float* __restrict__ cbmax,
               FlagList flags, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  using namespace tcenc;
  extern __shared__ __align__(1024) char smem_raw[];
  char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  char* Atile = smem;
  char* Bbuf = Atile + kATile;
  float* sC = reinterpret_cast<float*>(Bbuf + 2 * kTcBTile);
  float2* sNL = reinterpret_cast<float2*>(sC + kChunk * kD);
  float* sNa = reinterpret_cast<float*>(sNL + kChunk);
  float* sRa = sNa + kChunk;  // [h][thread]
  float* sPm = sRa + 16 * kThreads;
  uint32_t* sMask = reinterpret_cast<uint32_t*>(sPm + 16 * kThreads);  // [32-column word][thread]
  __shared__ __align__(16) float sH[kD * kD];
  __shared__ __align__(8) uint64_t bar_b, bar_mma;
  __shared__ uint32_t tmem_slot;

  const int tid = threadIdx.x, warp = tid >> 5;
  const int64_t g = g_begin + blockIdx.y;
  const int64_t G_range = gridDim.y;
  const int64_t i = (int64_t)blockIdx.x * kThreads + tid;
  const bool live = i < set.M;
  const int64_t vi = live ? i * G_range + (g - g_begin) : 0;
  const CbView cw = cbs.cb[sd.st[sd.s]];
  const int nchunk = (cw.K + kTcCols - 1) / kTcCols;  // 1 or 2
  const int S = sd.S, B = sd.B;
  const float cmul = bound_mult(n_fixed + sd.s);

  if (tid < kD * kD) sH[tid] = set.Hb[g * kD * kD + tid];
  if (warp == 0) tc::tmem_alloc(&tmem_slot, 2 * kTcCols);
  if (tid == 0) {
    tc::mbar_init(tc::smem_u32(&bar_b), 1);
    tc::mbar_init(tc::smem_u32(&bar_mma), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  if (tid == 0) {  // this group's B images, one bulk copy per 128-codeword chunk
    tc::mbar_expect_tx(tc::smem_u32(&bar_b), (uint32_t)(nchunk * kTcBTile));
    for (int c = 0; c < nchunk; ++c)
      tc::bulk_copy_g2s(tc::smem_u32(Bbuf + c * kTcBTile),
                        bimg + ((size_t)(g - g_begin) * nchunk + c) * kTcBTile, kTcBTile,
                        tc::smem_u32(&bar_b));
  }
  stage_chunk(cw.C, 0, cw.K, sH, cmul, sC, sNL, sNa);
  __syncthreads();

  // Na <= max row sum of |H_g| * L1max * cinf over the codebook (cbmax: L1max, cinf)
  float hrow = 0.f;
#pragma unroll
  for (int a = 0; a < kD; ++a) {
    float rs = 0.f;
#pragma unroll
    for (int b = 0; b < kD; ++b) rs += fabsf(sH[a * kD + b]);
    hrow = fmaxf(hrow, rs);
  }
  const float l1max = cbmax[0], cinf = cbmax[1];
  const float na_max = hrow * l1max * cinf * (1.f + kU * cmul) * 1.0001f;
  constexpr uint32_t idesc = tc::idesc_tf32(kRows, kTcCols);

  const int Bh = (sd.s == 0) ? 1 : (live ? bb.n_in[vi] : 1);
  const int Bmax = (sd.s == 0) ? 1 : B;  // uniform hypothesis loop bound of the CTA
  float th[kD], tl[kD];
  if (live) {
    dfl::target(set, cbs, n_fixed, i, g, th, tl, err);
  } else {
#pragma unroll
    for (int j = 0; j < kD; ++j) th[j] = tl[j] = 0.f;
  }
  // The sorted top-L list in registers. An insertion compares with every entry at once and moves
  // each by at most one place (no chain along the list): about 45 instructions, run only when some
  // lane's candidate enters. (A shifting insert in shared memory took a dependent load, compare and
  // store per place.)
  float topv[L];
  int topi[L];
#pragma unroll
  for (int j = 0; j < L; ++j) {
    topv[j] = INFINITY;
    topi[j] = 0x7fffffff;
  }
  float tau_x = INFINITY;
  bool ok = true;
  const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
  // Terms of hypothesis h (zero for a thread without it) and its A row. The terms of h + 1
  // are computed while the tensor cores run the pass of h, its row written once that pass
  // has completed.
  auto hyp_terms = [&](int h, float m2q[kD], float& base, float& nbeta, float& eps) {
#pragma unroll
    for (int p = 0; p < kD; ++p) m2q[p] = 0.f;
    base = nbeta = eps = 0.f;
    if (live && h < Bh) {
      float rh[kD], rl[kD], rr, ra, pmax;
      const int32_t* pc = bb.hyp_in ? bb.hyp_in + (vi * B + h) * S : nullptr;
      hyp_residual_pair(th, tl, cbs, sd, pc, rh, rl, err);
      hyp_terms_pair(rh, rl, sH, m2q, rr, ra, pmax);
      sRa[h * kThreads + tid] = ra;
      sPm[h * kThreads + tid] = pmax;
      base = rr - kU * cmul * ra;
      nbeta = -2.f * kU * cmul * pmax;
      eps = 1.52587890625e-05f *  // 2^-16
            (fabsf(base) + na_max + 2.f * pmax * l1max * 1.0001f + fabsf(nbeta) * l1max);
    }
  };
  auto write_a = [&](const float m2q[kD], float base, float nbeta) {
    uint32_t row[kK];
#pragma unroll
    for (int p = 0; p < kD; ++p) {
      uint32_t hh, ll;
      split(m2q[p], hh, ll);
      row[p] = hh;
      row[8 + p] = hh;
      row[16 + p] = ll;
    }
    const uint32_t one = __float_as_uint(1.f);
    row[24] = one;
    row[25] = one;
    split(nbeta, row[26], row[28]);
    row[27] = row[26];
    split(base, row[29], row[30]);
    row[31] = 0u;
    put_row(Atile, tid, row);
  };
  float m2q[kD], base, nbeta, eps;
  hyp_terms(0, m2q, base, nbeta, eps);
  write_a(m2q, base, nbeta);
  for (int h = 0; h < Bmax && ok; ++h) {
    const bool act = live && h < Bh;
    tc::fence_async_smem();
    tc::tc_fence_before();
    __syncthreads();
    if (tid == 0) {
      bool bok = true;
      if (h == 0) bok = tc::mbar_wait(tc::smem_u32(&bar_b), 0u, err);
      if (bok) {
        tc::tc_fence_after();
        const uint32_t a0 = tc::smem_u32(Atile);
        for (int c = 0; c < nchunk; ++c) {
          const uint32_t b0 = tc::smem_u32(Bbuf + c * kTcBTile);
#pragma unroll
          for (int ks = 0; ks < kK / 8; ++ks)
            tc::mma_tf32(tmem + (uint32_t)(c * kTcCols),
                         tc::smem_desc(a0 + ks * 256, 128, (kK / 4) * 128),
                         tc::smem_desc(b0 + ks * 256, 128, (kK / 4) * 128), idesc,
                         ks > 0 ? 1u : 0u);
        }
        tc::mma_commit(tc::smem_u32(&bar_mma));
      } else {
        tc::mbar_arrive(tc::smem_u32(&bar_mma));  // release the waiters; ok turns false
      }
      if (!bok) raise_error(err, ERRBIT_TIMEOUT);
    }
    float nm2q[kD], nbase, nnbeta, neps;
    if (h + 1 < Bmax) hyp_terms(h + 1, nm2q, nbase, nnbeta, neps);
    bool wok = tc::mbar_wait(tc::smem_u32(&bar_mma), (uint32_t)(h & 1), err);
    if (h == 0 && tid == 0) wok = wok && tc::mbar_try_wait(tc::smem_u32(&bar_b), 0u);
    ok = __syncthreads_and(wok);
    if (!ok) break;
    tc::tc_fence_after();

    const int nq = nchunk * 2;  // 64-column loads
    if (h == 0) {  // tau from the block minima of y for hypothesis 0
      float bl[L];
#pragma unroll
      for (int j = 0; j < L; ++j) bl[j] = INFINITY;
#pragma unroll 1
      for (int q = 0; q < nq; ++q) {
        uint32_t v[64];
        tc::tmem_ld64_wait(trow + 64 * q, v);
#pragma unroll
        for (int b4 = 0; b4 < 4; ++b4) {
          float m = __uint_as_float(v[16 * b4]);
#pragma unroll
          for (int e = 1; e < 16; ++e) m = fminf(m, __uint_as_float(v[16 * b4 + e]));
          m = (m == m) ? m : INFINITY;  // a block of NaNs holds no bound
#pragma unroll
          for (int j = 0; j < L; ++j) {
            const float t = fmaxf(bl[j], m);
            bl[j] = fminf(bl[j], m);
            m = t;
          }
        }
      }
      if (act) tau_x = __fadd_ru(bl[L - 1], eps);
    }
    // Candidates of hypothesis h: masks of all its columns first (a subtraction and a funnel shift per
    // score), then their members in codeword order, scored again with the fast stage's chain and
    // inserted. A warp's lanes walk their own masks side by side: it takes as many rounds as its longest
    // list of about five, where rounds per 32 columns took three times as many (three stages over 11008 x
    // 11 vectors 548 -> 512 us). The threshold is that of the pass's start (-inf for a thread without
    // this hypothesis).
    const float thrD = act ? __fadd_ru(fminf(topv[L - 1], tau_x), eps) : -INFINITY;
    // y <= thrD as the sign of y - (the next number above thrD): one instruction on the FMA pipe and
    // one on the ALU pipe, which had both of the compare form
    const float up = thrD < INFINITY && thrD > -INFINITY
                         ? __int_as_float(__float_as_int(thrD) +
                                          (thrD > 0.f ? 1 : thrD < 0.f ? -1 : 0)) +
                               (thrD == 0.f ? 1.401298464e-45f : 0.f)
                         : thrD;
    uint32_t words = 0u;  // the mask words with members
#pragma unroll 1
    for (int q = 0; q < nq; ++q) {
      uint32_t v[64];
      tc::tmem_ld64_wait(trow + 64 * q, v);
      uint32_t part[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int e = 15; e >= 0; --e)
#pragma unroll
        for (int w = 0; w < 4; ++w)
          part[w] = __funnelshift_l(__float_as_uint(__fsub_rn(__uint_as_float(v[16 * w + e]), up)),
                                    part[w], 1);
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const int k0 = 64 * q + 32 * w;
        uint32_t m = part[2 * w] | part[2 * w + 1] << 16;
        if (k0 + 32 > cw.K)  // padding columns (only with an unbounded threshold)
          m &= k0 < cw.K ? (1u << (cw.K - k0)) - 1u : 0u;
        sMask[(2 * q + w) * kThreads + tid] = m;
        words |= m ? 1u << (2 * q + w) : 0u;
      }
    }
    int kw = 0;
    uint32_t m = 0u;
    while (m | words) {
      if (m == 0u) {
        const int w = __ffs(words) - 1;
        words &= words - 1u;
        m = sMask[w * kThreads + tid];
        kw = 32 * w;
      }
      const int k = kw + __ffs(m) - 1;
      m &= m - 1u;
      const float4 c0 = *reinterpret_cast<const float4*>(sC + k * kD);
      const float4 c1 = *reinterpret_cast<const float4*>(sC + k * kD + 4);
      const float2 nl = sNL[k];
      float sv = base + nl.x;
      sv = fmaf(m2q[0], c0.x, sv);
      sv = fmaf(m2q[1], c0.y, sv);
      sv = fmaf(m2q[2], c0.z, sv);
      sv = fmaf(m2q[3], c0.w, sv);
      sv = fmaf(m2q[4], c1.x, sv);
      sv = fmaf(m2q[5], c1.y, sv);
      sv = fmaf(m2q[6], c1.z, sv);
      sv = fmaf(m2q[7], c1.w, sv);
      sv = fmaf(nbeta, nl.y, sv);
      if (sv < topv[L - 1]) {  // insert before the first entry strictly above sv
        const int si = (h << 16) | k;
#pragma unroll
        for (int j = L - 1; j >= 0; --j) {
          const bool below = j > 0 && sv < topv[j > 0 ? j - 1 : 0];
          const bool here = sv < topv[j];
          topi[j] = below ? topi[j > 0 ? j - 1 : 0] : (here ? si : topi[j]);
          topv[j] = below ? topv[j > 0 ? j - 1 : 0] : (here ? sv : topv[j]);
        }
      }
    }
    __syncwarp();
    tc::tc_fence_before();
    if (h + 1 < Bmax) {  // the pass of h has completed: its A tile is free
      write_a(nm2q, nbase, nnbeta);
#pragma unroll
      for (int p = 0; p < kD; ++p) m2q[p] = nm2q[p];
      base = nbase;
      nbeta = nnbeta;
      eps = neps;
    }
  }
  // let the codebook copy land before the CTA ends (bounded), then free the tensor memory
  if (!ok && tid == 0) tc::mbar_wait(tc::smem_u32(&bar_b), 0u, err);
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 2 * kTcCols);
  beam_list_finish<L>(set, cbs, sd, bb, flags, live, i, g, vi, Bh, cmul, th, tl, sH, sNL, sNa, true,
                      sRa + tid, sPm + tid, kThreads, topv, topi, err);
}

// Exact stage for flagged vectors: one warp per vector; the lanes stride over the (h, k)
// candidates, re-score in fp32 pairs those whose fp32 lower bound is at most the vector's
// threshold (the keep-th exact err among the fast pass's listed candidates, which bounds
// every member of the exact top-Bs) and keep a sorted local top-Bs; a warp merge then
// extracts the global top-Bs in (err, h, k) order.
// Bound: latency (a few thousand vectors per stage). In fp64 the re-scoring alone kept an SM's
// fp64 pipe busy: 56 us per stage over 11008 x 11 vectors, now 31.
__global__ void __launch_bounds__(kThreads)
beam_stage_fallback_kernel(SetView set, int64_t g_begin, int64_t G_range, CbList cbs,
                           int n_fixed, StageDesc sd, BeamBufs bb, FlagList flags,
                           const float4* __restrict__ terms, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  __shared__ int queue[kThreads / 32][32], queue_h[kThreads / 32][32];
  const int lane = threadIdx.x & 31;
  int* q = queue[threadIdx.x >> 5];
  int* qh = queue_h[threadIdx.x >> 5];
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const unsigned cnt = min((unsigned long long)*flags.count, (unsigned long long)flags.cap);
  if (flags.total && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(flags.total, cnt);
  const int S = sd.S, B = sd.B, Bs = sd.Bs;
  const CbView cw = cbs.cb[sd.st[sd.s]];
  for (int64_t f = warp; f < cnt; f += nwarps) {
    const int64_t vi = flags.vec[f];
    const int64_t i = vi / G_range, g = g_begin + vi % G_range;
    const float* H = set.Hb + g * kD * kD;
    float th[kD], tl[kD];
    dfl::target(set, cbs, n_fixed, i, g, th, tl, err);
    const int Bh = (sd.s == 0) ? 1 : bb.n_in[vi];
    const float thr = flags.thr[f];
    const float cmul = bound_mult(n_fixed + sd.s);
    float be[16], bl[16];  // err pairs
    int bh[16], bk[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      be[j] = INFINITY;
      bl[j] = 0.f;
    }
    int nb = 0;
    // Candidates (h, k) are queued in increasing (h, k) order and scored one per lane, so
    // every lane still sees its own candidates in increasing (h, k): strict comparison in
    // the insertion keeps ties in (h, k) order.
    int qn = 0;
    auto drain = [&]() {
      __syncwarp();
      if (lane < qn) {
        const int h = qh[lane], k = q[lane];
        float rh[kD], rl[kD], c[kD], e, el;
        const int32_t* pc = bb.hyp_in ? bb.hyp_in + (vi * B + h) * S : nullptr;
        hyp_residual_pair(th, tl, cbs, sd, pc, rh, rl, err);
        load_vec(cw.C + (int64_t)k * kD, c);
        dfl::quad_err<true>(rh, rl, c, H, e, el);
        auto before = [&](int at) { return e < be[at] || (e == be[at] && el < bl[at]); };
        if (nb < Bs || before(nb - 1)) {
          int pos = nb < Bs ? nb : Bs - 1;
          while (pos > 0 && before(pos - 1)) {
            be[pos] = be[pos - 1];
            bl[pos] = bl[pos - 1];
            bh[pos] = bh[pos - 1];
            bk[pos] = bk[pos - 1];
            --pos;
          }
          be[pos] = e;
          bl[pos] = el;
          bh[pos] = h;
          bk[pos] = k;
          if (nb < Bs) ++nb;
        }
      }
      __syncwarp();
      qn = 0;
    };
    for (int h = 0; h < Bh; ++h) {
      float rh[kD], rl[kD];
      const int32_t* pc = bb.hyp_in ? bb.hyp_in + (vi * B + h) * S : nullptr;
      hyp_residual_pair(th, tl, cbs, sd, pc, rh, rl, err);
      float m2q[kD], rr, ra, pmax;
      hyp_terms_pair(rh, rl, H, m2q, rr, ra, pmax);
      const float base = rr - kU * cmul * ra;
      const float nbeta = -2.f * kU * cmul * pmax;
      for (int k0 = 0; k0 < cw.K; k0 += 32) {
        const int k = k0 + lane;
        bool cand = false;
        if (k < cw.K) {
          float c[kD], n, na, l1;
          load_vec(cw.C + (int64_t)k * kD, c);
          if (terms) {  // the tensor-core stage's codeword terms of the group
            const float4 t = terms[(g - g_begin) * cw.K + k];
            n = t.x;
            na = t.y;
            l1 = t.z;
          } else {
            codeword_terms(c, H, n, na, l1);
          }
          cand = base + low_from(n, na, l1, c, m2q, nbeta, cmul) <= thr;
        }
        const unsigned m = __ballot_sync(0xffffffffu, cand);
        const int n = __popc(m);
        if (qn + n > 32) drain();
        if (cand) {
          const int pos = qn + __popc(m & ((1u << lane) - 1u));
          q[pos] = k;
          qh[pos] = h;
        }
        qn += n;
      }
    }
    drain();
    // Warp merge: rounds of (min over the lanes' heads by (err, h, k)); the winner pops.
    int head = 0;
    int32_t* out = bb.hyp_out + vi * B * S;
    const int total = (int)min((int64_t)Bs, (int64_t)Bh * cw.K);
    for (int j = 0; j < total; ++j) {
      float e = head < nb ? be[head] : INFINITY, el = head < nb ? bl[head] : 0.f;
      int hh = head < nb ? bh[head] : 0x7fffffff;
      int kk = head < nb ? bk[head] : 0x7fffffff;
      int src = lane;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const float oe = __shfl_xor_sync(0xffffffffu, e, off);
        const float ol = __shfl_xor_sync(0xffffffffu, el, off);
        const int oh = __shfl_xor_sync(0xffffffffu, hh, off);
        const int ok = __shfl_xor_sync(0xffffffffu, kk, off);
        const int os = __shfl_xor_sync(0xffffffffu, src, off);
        const bool take =
            oe < e || (oe == e && (ol < el || (ol == el && (oh < hh || (oh == hh && ok < kk)))));
        if (take) {
          e = oe;
          el = ol;
          hh = oh;
          kk = ok;
          src = os;
        }
      }
      if (lane == src) ++head;
      if (lane == 0) {
        if (hh >= Bh || kk >= cw.K) {
          raise_error(err, ERRBIT_NUMERIC);
          hh = 0;
          kk = 0;
        }
        const int32_t* pc = bb.hyp_in ? bb.hyp_in + (vi * B + hh) * S : nullptr;
        for (int q = 0; q < sd.s; ++q) out[j * S + q] = pc[q];
        out[j * S + sd.s] = kk;
      }
    }
    if (lane == 0) bb.n_out[vi] = total;
  }
}

// fp32 err of a whole tuple for vector (i, g): the fixed codebooks' codes, then for each
// searched stage q the code sc[q] (or, with sc null, the code already stored), with a bound
// on its distance from the exact err: the residual's rounding (m subtractions) and the two
// FMA chains of the quadratic form stay below (16 + 2 m) u a^T |H| a, a_j = |t_j| + sum of
// the |c_j| subtracted; the bound uses the multiplier of the score bounds, about twice that.
__device__ void tuple_err32(const SetView& set, const CbList& cbs, int n_fixed,
                            const StageDesc& sd, int64_t i, int64_t g, const int32_t* sc,
                            const float* H, float& e, float& bnd, unsigned* err) {
  float r[kD], a[kD];
  target32(set, cbs, n_fixed, i, g, r, a, err);
  for (int q = 0; q < sd.S; ++q) {
    const CbView& cb = cbs.cb[sd.st[q]];
    const int32_t k = sc ? sc[q] : cb.codes[i * cb.ld + g];
    if (!code_ok(k, cb.K, err)) continue;
    float c[kD];
    load_vec(cb.C + (int64_t)k * kD, c);
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      r[j] -= c[j];
      a[j] += fabsf(c[j]);
    }
  }
  float ee = 0.f, na = 0.f;
#pragma unroll
  for (int b = 0; b < kD; ++b) {
    float hb = 0.f, hab = 0.f;
#pragma unroll
    for (int a2 = 0; a2 < kD; ++a2) {
      hb = fmaf(r[a2], H[a2 * kD + b], hb);
      hab = fmaf(a[a2], fabsf(H[a2 * kD + b]), hab);
    }
    ee = fmaf(hb, r[b], ee);
    na = fmaf(hab, a[b], na);
  }
  e = ee;
  bnd = kU * bound_mult(n_fixed + sd.S + 1) * na;
}

// err of a whole tuple of vector (i, g) in fp64: the fixed codebooks' codes, then for each searched
// stage q the code sc[q] (with sc null: the code already stored).
__device__ double tuple_err64(const SetView& set, const CbList& cbs, int n_fixed,
                              const StageDesc& sd, int64_t i, int64_t g, const int32_t* sc,
                              const float* H, unsigned* err) {
  double r[kD];
  target64(set, cbs, n_fixed, i, g, r, err);
  for (int q = 0; q < sd.S; ++q) {
    const CbView& cb = cbs.cb[sd.st[q]];
    const int32_t k = sc ? sc[q] : cb.codes[i * cb.ld + g];
    if (!code_ok(k, cb.K, err)) continue;
    const float* c = cb.C + (int64_t)k * kD;
#pragma unroll
    for (int j = 0; j < kD; ++j) r[j] -= (double)c[j];
  }
  return quad_err64(r, nullptr, H);
}

// The same err in fp32 pairs (GB300's fp64 pipe made it most of the kernel's time): within a few 2^-48
// of |d|^T |H| |d| for the tuple's residual d, itself known to 2^-48 of the terms that it is left over
// from, so its fp32 rounding is fp64's but for the last place now and then. An err beyond fp32, and one
// so small that products lose their low parts (TwoProduct is exact above about 2^-102), are
// evaluated in fp64.
__device__ __forceinline__ float tuple_err_pair(const SetView& set, const CbList& cbs, int n_fixed,
                                                const StageDesc& sd, int64_t i, int64_t g,
                                                const int32_t* sc, const float* H, unsigned* err) {
  constexpr float kSmallest = 7.8886091e-31f;  // 2^-100
  float rh[kD], rl[kD], zero[kD], eh, el;
  dfl::target(set, cbs, n_fixed, i, g, rh, rl, err);
#pragma unroll
  for (int j = 0; j < kD; ++j) zero[j] = 0.f;
  for (int q = 0; q < sd.S; ++q) {
    const CbView& cb = cbs.cb[sd.st[q]];
    const int32_t k = sc ? sc[q] : cb.codes[i * cb.ld + g];
    if (!code_ok(k, cb.K, err)) continue;
    float c[kD];
    load_vec(cb.C + (int64_t)k * kD, c);
#pragma unroll
    for (int j = 0; j < kD; ++j) {
      float sj, ej;
      dfl::two_sum(rh[j], -c[j], sj, ej);
      rh[j] = sj;
      rl[j] = __fadd_rn(rl[j], ej);
    }
  }
  dfl::quad_err<true>(rh, rl, zero, H, eh, el);
  const float e = __fadd_rn(eh, el);
  if (e >= kSmallest && e <= 3.402823466e38f) return e;
  bool exact = true;  // an exact tuple: the err is 0
#pragma unroll
  for (int j = 0; j < kD; ++j) exact = exact && rh[j] == 0.f && rl[j] == 0.f;
  return exact ? 0.f : (float)tuple_err64(set, cbs, n_fixed, sd, i, g, sc, H, err);
}

// Final step of a multi-stage (or keep-if-better) encode: write the best tuple, or keep the
// tuple already in the codes when its err is strictly smaller. The comparison is decided by
// fp32 errs with bounds when they separate, in fp64 otherwise; an unchanged tuple needs no
// comparison. vec_err (optional) is the err of the tuple kept.
__global__ void beam_finalize_kernel(SetView set, int64_t g_begin, int64_t G_range,
                                     CbList cbs, int n_fixed, StageDesc sd,
                                     const int32_t* __restrict__ hyp, bool keep_if_better,
                                     float* __restrict__ vec_err, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const int64_t nvec = set.M * G_range;
  const int S = sd.S, B = sd.B;
  for (int64_t vi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; vi < nvec;
       vi += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = vi / G_range, g = g_begin + vi % G_range;
    const float* H = set.Hb + g * kD * kD;
    const int32_t* best = hyp + vi * B * S;
    bool use_old = false;
    bool exact = false;
    if (keep_if_better) {
      bool same = true;
      for (int q = 0; q < S; ++q) {
        const CbView& cb = cbs.cb[sd.st[q]];
        same = same && cb.codes[i * cb.ld + g] == best[q];
      }
      if (!same) {
        float en, bn, eo, bo;
        tuple_err32(set, cbs, n_fixed, sd, i, g, best, H, en, bn, err);
        tuple_err32(set, cbs, n_fixed, sd, i, g, nullptr, H, eo, bo, err);
        if (eo + bo < en - bn) {
          use_old = true;
        } else if (!(eo - bo >= en + bn)) {
          exact = true;  // not separated (or not finite): decide in fp64
        }
      }
    }
    if (exact) {
      const double e_new = tuple_err64(set, cbs, n_fixed, sd, i, g, best, H, err);
      use_old = tuple_err64(set, cbs, n_fixed, sd, i, g, nullptr, H, err) < e_new;
    }
    if (vec_err)
      vec_err[i * set.G_sub + g] =
          tuple_err_pair(set, cbs, n_fixed, sd, i, g, use_old ? nullptr : best, H, err);
    if (!use_old) {
      for (int q = 0; q < S; ++q) {
        const CbView& cb = cbs.cb[sd.st[q]];
        cb.codes[i * cb.ld + g] = best[q];
      }
    }
  }
}

// err of the tuple currently in the codes (all covering codebooks), in fp32 pairs.
__global__ void residual_err_kernel(SetView set, int64_t g_begin, int64_t G_range, CbList cbs,
                                    float* __restrict__ vec_err, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const int64_t nvec = set.M * G_range;
  StageDesc none{};
  for (int64_t vi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; vi < nvec;
       vi += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = vi / G_range, g = g_begin + vi % G_range;
    vec_err[i * set.G_sub + g] = tuple_err_pair(set, cbs, cbs.n, none, i, g, nullptr,
                                                set.Hb + g * kD * kD, err);
  }
}

// --------------------------------------------------------------------------- k-means init
__global__ void kmeans_init_kernel(SetView set, CbList fixed, int K, uint64_t seed,
                                   float* __restrict__ C_out, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  const int64_t n = set.M * set.G_sub;
  // Stratum k of the vector index range: [floor(k n / K), floor((k+1) n / K)).
  const int64_t lo = (int64_t)(((uint64_t)k * (uint64_t)n) / (uint64_t)K);
  const int64_t hi = (int64_t)(((uint64_t)(k + 1) * (uint64_t)n) / (uint64_t)K);
  const int64_t v = lo + (int64_t)(splitmix64(seed, (uint64_t)k) % (uint64_t)(hi - lo));
  const int64_t i = v / set.G_sub, g = v % set.G_sub;
  double r[kD];
  target64(set, fixed, fixed.n, i, g, r, err);
#pragma unroll
  for (int j = 0; j < kD; ++j) C_out[(int64_t)k * kD + j] = (float)r[j];
}

}  // namespace

// =============================================================================== host side
template <class Kern>
static crvq_status set_smem_attr(Kern k, size_t bytes) {
  CRVQ_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  return CRVQ_OK;
}

crvq_status launch_kmeans_init(const SetView& set, const CbList& fixed, int K, uint64_t seed,
                               float* C_out, cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  ProfScope ps("kmeans_init", stream, (double)K);
  CRVQ_CUDA(launch_pdl(kmeans_init_kernel, dim3((unsigned)ceil_div(K, 128)), dim3(128), 0, stream,
                       set, fixed, K, seed, C_out, err));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

namespace {

template <int L>
crvq_status launch_beam_stage_L(const SetView& set, int64_t g_begin, int64_t G_range,
                                const CbList& cbs, int n_fixed, const StageDesc& sd,
                                const BeamBufs& bb, const FlagList& fl, unsigned* err,
                                double units, cudaStream_t stream) {
  dim3 grid((unsigned)ceil_div(set.M, kThreads), (unsigned)G_range);
  ProfScope ps("encode_beam_stage", stream, units);
  CRVQ_CUDA(launch_pdl(beam_stage_kernel<L>, grid, dim3(kThreads), 0, stream, set, g_begin, cbs,
                       n_fixed, sd, bb, fl, err));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

template <int L>
crvq_status launch_beam_tc_L(const SetView& set, int64_t g_begin, int64_t G_range,
                             const CbList& cbs, int n_fixed, const StageDesc& sd,
                             const BeamBufs& bb, const char* bimg, const float* cbmax,
                             const FlagList& fl, unsigned* err, double units,
                             cudaStream_t stream) {
  CRVQ_TRY(set_smem_attr(beam_tc_kernel<L>, kBeamTcSmem));
  dim3 grid((unsigned)ceil_div(set.M, kThreads), (unsigned)G_range);
  ProfScope ps("encode_beam_stage", stream, units);
  CRVQ_CUDA(launch_pdl(beam_tc_kernel<L>, grid, dim3(kThreads), kBeamTcSmem, stream, set, g_begin,
                       cbs, n_fixed, sd, bb, bimg, cbmax, fl, err));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

// The tensor-core stage for codebooks of at most 256 codewords and lists of at most 9 entries
// (beam width up to 8): B images of the stage codebook for the group range (prep_b with the
// stage's bound multiplier), then beam_tc_kernel. `work` holds beam_tc_scratch_bytes.
size_t beam_tc_scratch_bytes(int64_t G_range, int K) {
  const int nchunk = (int)ceil_div(K, kTcCols);
  return 256 + (size_t)G_range * nchunk * kTcBTile +
         align_up((size_t)G_range * K * sizeof(float4), 256) + 256;
}

// The codeword terms within that scratch.
float4* beam_tc_terms(char* work, int64_t G_range, int K) {
  return reinterpret_cast<float4*>(work + 256 +
                                   (size_t)G_range * ceil_div(K, kTcCols) * kTcBTile);
}

// CRVQ_BEAM_TC=0 in the environment (read at every call) keeps every stage on the SIMT kernel:
// the two forms give the same lists, which tests compare.
bool beam_tc_applies(const StageDesc& sd, const CbList& cbs, int64_t G_range) {
  const char* v = getenv("CRVQ_BEAM_TC");
  if (v && v[0] == '0') return false;
  const int K = cbs.cb[sd.st[sd.s]].K;
  return K <= 2 * kTcCols && sd.Bs + 1 <= 9 &&
         (size_t)G_range * ceil_div(K, kTcCols) * kTcBTile <= (size_t(256) << 20);
}

crvq_status launch_beam_stage_tc(const SetView& set, int64_t g_begin, int64_t G_range,
                                 const CbList& cbs, int n_fixed, const StageDesc& sd,
                                 const BeamBufs& bb, const FlagList& fl, unsigned* err,
                                 char* work, double units, cudaStream_t stream) {
  const CbView& cw = cbs.cb[sd.st[sd.s]];
  const int nchunk = (int)ceil_div(cw.K, kTcCols);
  float* cbmax = reinterpret_cast<float*>(work);
  char* bimg = work + 256;
  float4* tout = beam_tc_terms(work, G_range, cw.K);
  const float uc = kU * bound_mult(n_fixed + sd.s);
  {
    ProfScope pb("encode_prep_b", stream, (double)G_range * nchunk * kTcCols);
    CRVQ_CUDA(launch_pdl(prep_b_kernel, prep_b_grid(G_range, nchunk, sm_count()), dim3(128), 0, stream,
                         set, g_begin, cw.C, cw.K, nchunk, uc, bimg, tout, cbmax, fl.count));
    CRVQ_LAUNCHED();
  }
  // the list length L = Bs + 1, rounded up to an instantiated size
  auto go = [&](auto L) {
    return launch_beam_tc_L<decltype(L)::value>(set, g_begin, G_range, cbs, n_fixed, sd, bb,
                                                 bimg, cbmax, fl, err, units, stream);
  };
  const int need = sd.Bs + 1;
  if (need <= 2) return go(std::integral_constant<int, 2>{});
  if (need <= 3) return go(std::integral_constant<int, 3>{});
  if (need <= 5) return go(std::integral_constant<int, 5>{});
  return go(std::integral_constant<int, 9>{});
}

crvq_status launch_beam_stage(const SetView& set, int64_t g_begin, int64_t G_range,
                              const CbList& cbs, int n_fixed, const StageDesc& sd,
                              const BeamBufs& bb, const FlagList& fl, unsigned* err,
                              double units, cudaStream_t stream) {
  auto go = [&](auto L) {
    return launch_beam_stage_L<decltype(L)::value>(set, g_begin, G_range, cbs, n_fixed, sd, bb,
                                                   fl, err, units, stream);
  };
  const int need = sd.Bs + 1;
  if (need <= 2) return go(std::integral_constant<int, 2>{});
  if (need <= 3) return go(std::integral_constant<int, 3>{});
  if (need <= 5) return go(std::integral_constant<int, 5>{});
  if (need <= 9) return go(std::integral_constant<int, 9>{});
  return go(std::integral_constant<int, 17>{});
}

// Scratch of one arg-min pass: codebook maxima (256 B) | B images (the columns that all groups
// share, then those of G_sub groups) | codeword terms of G_sub groups | counts of the two open lists
// (256 B) | narrow list | wide list (vector ids and thresholds). Sub-ranges of groups whose images
// and terms take at most 256 MB.
struct ArgminLayout {
  int nchunk;
  int64_t G_sub;
  size_t bbytes, tbytes, obytes, fbytes, total;
};

ArgminLayout argmin_layout(int64_t M, int64_t G_range, int K) {
  ArgminLayout L{};
  if (K <= kSmallK) return L;  // argmin_small_kernel takes none
  L.nchunk = (int)ceil_div(K, kTcCols);
  const int64_t per_group = (int64_t)L.nchunk * kBCol + (int64_t)K * (int64_t)sizeof(float4);
  L.G_sub = std::max<int64_t>(1, std::min<int64_t>(G_range, (int64_t(256) << 20) / per_group));
  L.bbytes = (size_t)L.nchunk * kTcBTile + (size_t)L.G_sub * L.nchunk * kBCol;
  L.tbytes = align_up((size_t)L.G_sub * K * sizeof(float4), 256);
  L.obytes = align_up((size_t)M * L.G_sub * sizeof(NarrowRow), 256);
  L.fbytes = align_up((size_t)M * L.G_sub * (sizeof(int64_t) + sizeof(float)), 256);
  L.total = 256 + L.bbytes + L.tbytes + 256 + L.obytes + L.fbytes;
  return L;
}

// One arg-min pass over the groups [g_begin, g_begin + G_range): codebook s_idx searched, those
// before n_fixed fixed, codes to out unless it is null (with the statistics of st when it has any).
struct ArgminCall {
  int64_t g_begin, G_range;
  int n_fixed, s_idx;
  int32_t* out;
  int64_t out_ld, out_g0;
  StatsView st;
};

// Codebooks of at most 256 codewords: one persistent kernel, two CTAs per SM.
crvq_status launch_argmin_small(const SetView& set, const CbList& cbs, const ArgminCall& a,
                                const EncodeExtras& ex, unsigned* err, cudaStream_t stream) {
  const int64_t pairs = a.G_range * ceil_div(set.M, (int64_t)2 * tcenc::kRows);
  CRVQ_TRY(smem_limit((const void*)argmin_small_kernel, kArgminSmem));
  ProfScope ps(a.st.cnt ? "encode_argmin_lloyd" : "encode_argmin", stream,
               (double)set.M * a.G_range * cbs.cb[a.s_idx].K);
  CRVQ_CUDA(launch_pdl(argmin_small_kernel, dim3((unsigned)std::min<int64_t>(2 * sm_count(), pairs)),
                       dim3(256), kArgminSmem, stream, set, a.g_begin, a.G_range, cbs, a.n_fixed,
                       a.s_idx, a.out, a.out_ld, a.out_g0, ex.flag_total, a.st, ex.rowterms, err));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

// Larger codebooks: groups in sub-ranges (argmin_layout); per sub-range: images + per-group codeword
// terms (prep_b_split, which also writes the shared images and the codebook maxima the first time),
// the arg-min pass, and the exact decision of flagged rows.
crvq_status launch_argmin_large(const SetView& set, const CbList& cbs, const ArgminCall& a,
                                const EncodeExtras& ex, unsigned* err, cudaStream_t stream) {
  const int64_t g_begin = a.g_begin, G_range = a.G_range, out_ld = a.out_ld, out_g0 = a.out_g0;
  const int n_fixed = a.n_fixed, s_idx = a.s_idx, nsm = sm_count();
  int32_t* out = a.out;
  const StatsView& st = a.st;
  const CbView& cw = cbs.cb[s_idx];
  const ArgminLayout AL = argmin_layout(set.M, G_range, cw.K);
  const int nchunk = AL.nchunk;
  const int64_t G_sub = AL.G_sub;
  const size_t bbytes = AL.bbytes, tbytes = AL.tbytes;
  Scratch bmem;
  char* wbase = ex.work;
  if (!wbase || ex.work_bytes < AL.total) {
    CRVQ_TRY(bmem.alloc(AL.total, stream));
    wbase = bmem.as<char>();
  }
  float* cbmax = reinterpret_cast<float*>(wbase);
  char* bimg = wbase + 256;
  char* bgrp = bimg + (size_t)nchunk * kTcBTile;
  float4* tout = reinterpret_cast<float4*>(bimg + bbytes);
  FlagList fl;
  fl.count = reinterpret_cast<unsigned*>(wbase + 256 + bbytes + tbytes);
  const NarrowList nl{reinterpret_cast<NarrowRow*>(wbase + 256 + bbytes + tbytes + 256), fl.count + 1,
                      fl.total = ex.flag_total};
  fl.vec = reinterpret_cast<int64_t*>(wbase + 256 + bbytes + tbytes + 256 + AL.obytes);
  fl.cap = set.M * G_sub;
  fl.thr = reinterpret_cast<float*>(fl.vec + fl.cap);
  const float uc = kU * (tcenc::kCmul + 4.f * n_fixed);
  CRVQ_TRY(smem_limit((const void*)argmin_tc_kernel<true>, argmin_stream_smem(true)));
  CRVQ_TRY(smem_limit((const void*)argmin_tc_kernel<false>, argmin_stream_smem(false)));
  for (int64_t gs = g_begin; gs < g_begin + G_range; gs += G_sub) {
    const int64_t gn = std::min<int64_t>(G_sub, g_begin + G_range - gs);
    const int64_t nv = set.M * gn;
    fl.cap = nv;
    fl.thr = reinterpret_cast<float*>(fl.vec + nv);  // the count is cleared by prep_b
    {
      ProfScope pb("encode_prep_b", stream, (double)gn * nchunk * kTcCols);
      CRVQ_CUDA(launch_pdl(prep_b_split_kernel, prep_b_grid(gn, nchunk, nsm), dim3(128), 0, stream, set,
                           gs, cw.C, cw.K, nchunk, uc, gs == g_begin, bimg, bgrp, tout, cbmax, fl.count));
      CRVQ_LAUNCHED();
    }
    {
      // A tile per half (OWN) for codebooks of few chunks when every half on the chip gets one, a shared
      // tile otherwise. OWN / shared: 300 codewords, 12000 x 512 vectors 596 / 841 us, 1024 x 128 29 / 34;
      // 1024, 3001 x 371 249 / 296; 2048, 300 x 1000 206 / 204; 65536, 1024 x 1376 19.2 / 17.5 ms; one
      // tile per group (1024, 128 x 1024) 78 / 72 us; few groups (1024, 700 x 30) 36 / 33 us.
      const int64_t row_tiles = ceil_div(set.M, tcenc::kRows);
      const bool own = cw.K <= 2048 && row_tiles >= 2 && gn * row_tiles >= 4 * (int64_t)nsm;
      // row tiles per CTA: about sixteen waves of two CTAs per SM (a fine-grained tail)
      const int64_t per_group =
          std::max<int64_t>(1, (own ? 16 : 32) * (int64_t)nsm / std::max<int64_t>(1, gn));
      const int tiles = (int)std::max<int64_t>(own ? 2 : 1, ceil_div(row_tiles, per_group));
      const dim3 grid((unsigned)ceil_div(row_tiles, tiles), (unsigned)gn);
      ProfScope ps(st.cnt ? "encode_argmin_lloyd" : "encode_argmin", stream,
                   (double)nv * cw.K);
      auto* kernel = own ? argmin_tc_kernel<true> : argmin_tc_kernel<false>;
      CRVQ_CUDA(launch_pdl(kernel, grid, dim3(256), argmin_stream_smem(own), stream, set, gs,
                           cbs, n_fixed, s_idx, out, out_ld, out_g0, fl, nl, st, cbmax, bimg, bgrp, tout,
                           ex.rowterms, tiles, err));
      CRVQ_LAUNCHED();
    }
    {
      ProfScope pf("encode_exact", stream, 0.0);
      // few wide rows go to blocks, one each (eight per block of that grid at most)
      const unsigned blocks = (unsigned)std::min<int64_t>(nv, 2 * nsm);
      const unsigned many = cw.K <= kExactWarpK ? 0u : 8 * blocks;
      CRVQ_CUDA(launch_pdl(argmin_exact_warp_kernel,
                           dim3((unsigned)std::min<int64_t>(ceil_div(nv, 4), 16 * nsm)), dim3(128), 0,
                           stream, set, gs, gn, cbs, n_fixed, s_idx, out, out_ld, out_g0, nl, fl, many,
                           st, tout, err));
      if (many) {
        CRVQ_LAUNCHED();
        CRVQ_CUDA(launch_pdl(argmin_exact_kernel, dim3(blocks), dim3(kExactThreads), 0, stream, set, gs,
                             gn, cbs, n_fixed, s_idx, out, out_ld, out_g0, fl, many, st, tout, err));
      }
      CRVQ_LAUNCHED();
    }
  }
  return CRVQ_OK;
}

// One range of groups [g_begin, g_begin + G_range) whose searched stages are sd.st[0..S).
crvq_status encode_range(const SetView& set, int64_t g_begin, int64_t G_range,
                         const CbList& cbs, int n_fixed, StageDesc sd, bool keep_if_better,
                         float* vec_err, const EncodeExtras& ex, unsigned* err,
                         cudaStream_t stream) {
  const int64_t nvec = set.M * G_range;
  if (nvec == 0) return CRVQ_OK;
  const int nsm = sm_count();
  const unsigned fin_blocks = (unsigned)std::min<int64_t>(ceil_div(nvec, 128), 8 * nsm);
  if (sd.S == 0) {
    if (vec_err) {
      CRVQ_CUDA(launch_pdl(residual_err_kernel, dim3(fin_blocks), dim3(128), 0, stream, set,
                           g_begin, G_range, cbs, vec_err, err));
      CRVQ_LAUNCHED();
    }
    return CRVQ_OK;
  }
  if (sd.S == 1) {
    // Arg-min over one codebook (the k-means assignment step). Written in place unless the
    // old code may be kept, in which case into a scratch tuple buffer that the finalize step
    // compares with the old tuple.
    const int s_idx = sd.st[0];
    const CbView& cw = cbs.cb[s_idx];
    Scratch tup_mem;
    int32_t* out = cw.codes;
    int64_t out_ld = cw.ld, out_g0 = 0;
    if (keep_if_better) {
      CRVQ_TRY(tup_mem.alloc((size_t)nvec * sizeof(int32_t), stream));
      out = tup_mem.as<int32_t>();
      out_ld = G_range;
      out_g0 = g_begin;
    }
    StatsView st{};
    if (ex.stats && !keep_if_better) st = *ex.stats;
    if (ex.discard_codes && !keep_if_better && !vec_err) out = nullptr;
    const ArgminCall ac{g_begin, G_range, n_fixed, s_idx, out, out_ld, out_g0, st};
    if (cw.K <= kSmallK)
      CRVQ_TRY(launch_argmin_small(set, cbs, ac, ex, err, stream));
    else
      CRVQ_TRY(launch_argmin_large(set, cbs, ac, ex, err, stream));
    if (ex.scores) *ex.scores += (double)nvec * cw.K;
    if (keep_if_better) {
      ProfScope ps3("encode_finalize", stream, 0.0);
      StageDesc one = sd;
      one.B = 1;
      one.Bs = 1;
      CRVQ_CUDA(launch_pdl(beam_finalize_kernel, dim3(fin_blocks), dim3(128), 0, stream, set,
                           g_begin, G_range, cbs, n_fixed, one, out, true, vec_err, err));
      CRVQ_LAUNCHED();
    } else if (vec_err) {
      ProfScope ps3("encode_finalize", stream, 0.0);
      CRVQ_CUDA(launch_pdl(residual_err_kernel, dim3(fin_blocks), dim3(128), 0, stream, set,
                           g_begin, G_range, cbs, vec_err, err));
      CRVQ_LAUNCHED();
    }
    return CRVQ_OK;
  }

  Scratch flag_mem;
  const size_t fl_bytes = (size_t)nvec * (sizeof(int64_t) + sizeof(float)) + 256;
  CRVQ_TRY(flag_mem.alloc(fl_bytes, stream));
  FlagList fl;
  fl.count = flag_mem.as<unsigned>();
  fl.vec = reinterpret_cast<int64_t*>(flag_mem.as<char>() + 256);
  fl.thr = reinterpret_cast<float*>(fl.vec + nvec);
  fl.cap = nvec;
  fl.total = ex.flag_total;

  // Beam over S >= 2 stages: stage kernels over double-buffered hypothesis arrays.
  Scratch hyp_mem;
  const int B = sd.B, S = sd.S;
  const size_t hyp_elems = (size_t)nvec * B * S;
  CRVQ_TRY(hyp_mem.alloc(2 * (hyp_elems + nvec) * sizeof(int32_t), stream));
  int32_t* hypA = hyp_mem.as<int32_t>();
  int32_t* hypB = hypA + hyp_elems;
  int32_t* nA = hypB + hyp_elems;
  int32_t* nB = nA + nvec;
  const int32_t* in_h = nullptr;
  const int32_t* in_n = nullptr;
  int32_t* out_h = hypA;
  int32_t* out_n = nA;
  double sc = 0.0;
  int64_t parents = 1;
  // scratch of the tensor-core stages (B images and terms of one stage codebook)
  size_t tc_bytes = 0;
  for (int s = 0; s < S; ++s) {
    StageDesc d = sd;
    d.s = s;
    d.Bs = (s == S - 1) ? 1 : B;
    if (beam_tc_applies(d, cbs, G_range))
      tc_bytes = std::max(tc_bytes, beam_tc_scratch_bytes(G_range, cbs.cb[sd.st[s]].K));
  }
  Scratch tc_mem;
  if (tc_bytes) CRVQ_TRY(tc_mem.alloc(tc_bytes, stream));
  for (int s = 0; s < S; ++s) {
    sd.s = s;
    sd.Bs = (s == S - 1) ? 1 : B;  // only the best tuple of the last stage is used
    BeamBufs bb{in_h, in_n, out_h, out_n};
    const int K = cbs.cb[sd.st[s]].K;
    const bool tc_stage = beam_tc_applies(sd, cbs, G_range);
    if (!tc_stage)  // (prep_b_kernel clears it for the tensor-core stages)
      CRVQ_CUDA(cudaMemsetAsync(fl.count, 0, sizeof(unsigned), stream));
    if (tc_stage)
      CRVQ_TRY(launch_beam_stage_tc(set, g_begin, G_range, cbs, n_fixed, sd, bb, fl, err,
                                    tc_mem.as<char>(), (double)nvec * parents * K, stream));
    else
      CRVQ_TRY(launch_beam_stage(set, g_begin, G_range, cbs, n_fixed, sd, bb, fl, err,
                                 (double)nvec * parents * K, stream));
    {
      ProfScope ps("encode_beam_fallback", stream, 0.0);
      CRVQ_CUDA(launch_pdl(beam_stage_fallback_kernel, dim3(4 * nsm), dim3(kThreads), 0, stream,
                           set, g_begin, G_range, cbs, n_fixed, sd, bb, fl, tc_stage ?
                           beam_tc_terms(tc_mem.as<char>(), G_range, K) : nullptr, err));
      CRVQ_LAUNCHED();
    }
    sc += (double)nvec * parents * K;
    parents = std::min<int64_t>(B, parents * K);
    in_h = out_h;
    in_n = out_n;
    out_h = (out_h == hypA) ? hypB : hypA;
    out_n = (out_n == nA) ? nB : nA;
  }
  if (ex.scores) *ex.scores += sc;
  ProfScope ps("encode_finalize", stream, 0.0);
  CRVQ_CUDA(launch_pdl(beam_finalize_kernel, dim3(fin_blocks), dim3(128), 0, stream, set, g_begin,
                       G_range, cbs, n_fixed, sd, in_h, keep_if_better, vec_err, err));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

}  // namespace

crvq_status launch_row_terms(const SetView& set, const CbList& cbs, int n_fixed, float4* rt,
                             const StatsView* st, cudaStream_t stream) {
  const int64_t nvec = set.M * set.G_sub;
  if (nvec == 0) return CRVQ_OK;
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(nvec, 128), 16 * sm_count());
  CRVQ_CUDA(launch_pdl(row_terms_kernel, dim3(blocks), dim3(128), 0, stream, set, cbs, n_fixed,
                       rt, st ? *st : StatsView{}, err));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

size_t argmin_scratch_bytes(int64_t M, int64_t G_range, int K) {
  return argmin_layout(M, G_range, K).total;
}

crvq_status launch_encode_beam(const SetView& set, const CbList& cbs, int n_fixed, int B,
                               bool keep_if_better, float* vec_err, const EncodeExtras& ex,
                               cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  // Group ranges with the same set of covering searched codebooks: boundaries at every G_cov.
  std::vector<int64_t> cuts = {0, set.G_sub};
  for (int s = n_fixed; s < cbs.n; ++s)
    if (cbs.cb[s].G_cov > 0 && cbs.cb[s].G_cov < set.G_sub) cuts.push_back(cbs.cb[s].G_cov);
  std::sort(cuts.begin(), cuts.end());
  cuts.erase(std::unique(cuts.begin(), cuts.end()), cuts.end());
  if (ex.stats && cuts.size() > 2)
    return fail(CRVQ_ERR_UNSUPPORTED, "fused statistics need one group range");
  for (size_t r = 0; r + 1 < cuts.size(); ++r) {
    const int64_t g0 = cuts[r], g1 = cuts[r + 1];
    StageDesc sd{};
    sd.S = 0;
    sd.B = B;
    sd.Bs = B;
    for (int s = n_fixed; s < cbs.n; ++s)
      if (g0 < cbs.cb[s].G_cov) sd.st[sd.S++] = s;
    CRVQ_TRY(encode_range(set, g0, g1 - g0, cbs, n_fixed, sd, keep_if_better, vec_err, ex, err,
                          stream));
  }
  return CRVQ_OK;
}

}  // namespace crvq
