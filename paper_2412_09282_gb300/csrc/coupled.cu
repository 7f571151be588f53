// Code search under the full Alg. 1 loss (QuantLoss ||W X - W_enc X||^2 = tr(dW H dW^T)), with
// the cross-group terms that the block-diagonal search leaves out: a Gauss-Seidel sweep over
// the groups of one codebook, the others fixed (Sec. 3.1 codes; Alg. 1 QuantLoss).
//
// The loss separates over rows. For row i and group g, with every other group fixed,
//   L = D_g^T H_gg D_g + 2 D_g^T b_g + const,  b_g = sum_{g' != g} H_gg' D_g',  D = W - W_enc,
// and with D_g = t - c (t: the row segment minus the other codebooks' codewords) completing the
// square makes the best codeword the block-diagonal arg-min for the shifted target
//   t' = t + H_gg^-1 b_g,
// so each group step is an exact arg-min as the encode path decides it, on t'. Groups are visited
// in order, each with the current codes of the others, so the loss never rises.
//
// Blocked (lazy) evaluation of b_g: the channels are taken in blocks of 256 (32 groups). At
// the start of a block one tensor-core product gives B^T = H[block rows, :] D^T for the current
// D (256 x M); inside the block each group step adds its change dD_g H[g, g'] to the columns of
// the later groups g' of the block, and later blocks see the new D through their own product.
// Every b_g therefore includes every earlier decision of the sweep, as the sequential
// definition requires, with one product of 2 M N^2 flops per sweep in total. D_g is
// recomputed from W after each decision (in fp32 pairs, rounded once), so it does not drift.
//
// The rows do not see one another, so all 32 group steps of a block run in one kernel
// (coupled_block_kernel), a CTA carrying up to 32 rows through them with its slice of B^T in shared
// memory, and the launches between steps (five per group: target, operand images, arg-min, exact
// decisions, update) and the round trips of B^T through L2 are gone. Its scores run on the fp32 pipe, and
// a row that they leave open is a scan of the codebook by one warp, so for large codebooks and many rows
// the steps go through the encode path's tensor-core arg-min instead (coupled_target_kernel,
// launch_encode_beam on the shifted targets, coupled_apply_kernel): the same decisions, on the same t'.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "img.cuh"
#include "kernels.h"
#include "score.cuh"
#include "tc_ops.cuh"

namespace crvq {

namespace {

constexpr int kBlockCols = 256;                 // channels per lazy block (32 groups)
constexpr int kBlockG = kBlockCols / kD;

// (rh + rl) = vector (i, g) of W minus the codewords of every covering codebook but `which`.
__device__ __forceinline__ void others_target(const SetView& set, const CbList& cbs, int which,
                                              int64_t i, int64_t g, float rh[kD], float rl[kD],
                                              unsigned* err) {
  load_vec(set.T + i * set.ldT + g * kD, rh);
#pragma unroll
  for (int j = 0; j < kD; ++j) rl[j] = 0.f;
  for (int s = 0; s < cbs.n; ++s) {
    const CbView& cb = cbs.cb[s];
    if (s == which || g >= cb.G_cov) continue;
    const int32_t k = cb.codes[i * cb.ld + g];
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

// (rh + rl) - c, rounded once.
__device__ __forceinline__ float pair_minus(float rh, float rl, float c) {
  float s, e;
  dfl::two_sum(rh, -c, s, e);
  return __fadd_rn(s, __fadd_rn(rl, e));
}

// D = W - sum over the covering codebooks of C[code] (fp32 pairs, rounded once), M x N.
__global__ void __launch_bounds__(256)
residual_kernel(const float* __restrict__ W, int64_t M, int64_t N, CbList cbs, int which,
                float* __restrict__ D, unsigned* err) {
  const int64_t G = N / kD;
  const SetView set{W, N, M, G, nullptr};
  const CbView cw = cbs.cb[which];
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < M * G;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = v / G, g = v % G;
    float rh[kD], rl[kD], c[kD];
    others_target(set, cbs, which, i, g, rh, rl, err);
#pragma unroll
    for (int j = 0; j < kD; ++j) c[j] = 0.f;
    if (g < cw.G_cov) {
      const int32_t k = cw.codes[i * cw.ld + g];
      if (code_ok(k, cw.K, err)) load_vec(cw.C + (int64_t)k * kD, c);
    }
    float d[kD];
#pragma unroll
    for (int j = 0; j < kD; ++j) d[j] = pair_minus(rh[j], rl[j], c[j]);
    float* o = D + i * N + g * kD;
    *reinterpret_cast<float4*>(o) = make_float4(d[0], d[1], d[2], d[3]);
    *reinterpret_cast<float4*>(o + 4) = make_float4(d[4], d[5], d[6], d[7]);
  }
}

// Per group g < G_cov: the diagonal block H_gg of H (N x N) into Hb[g] (the arg-min's Hessian
// block) and its Cholesky factor, computed in fp64 and stored in fp32 (lower triangle, row
// major) with the reciprocals of its diagonal. One thread per group; a block without a factor
// reports ERRBIT_NUMERIC and gets a zero factor (its shifted targets are then not formed).
__global__ void __launch_bounds__(128)
block_factor_kernel(const float* __restrict__ H, int64_t N, int64_t G_cov,
                    float* __restrict__ Hb, float* __restrict__ Lf, float* __restrict__ Linv,
                    unsigned* err) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= G_cov) return;
  double L[kD * kD];
  bool ok = true;
  for (int r = 0; r < kD && ok; ++r)
    for (int c = 0; c <= r; ++c) {
      double sum = (double)H[(g * kD + r) * N + g * kD + c];
      for (int m = 0; m < c; ++m) sum -= L[r * kD + m] * L[c * kD + m];
      if (r == c) {
        if (!(sum > 0.0)) {
          ok = false;
          break;
        }
        L[r * kD + r] = sqrt(sum);
      } else {
        L[r * kD + c] = sum / L[c * kD + c];
      }
    }
  if (!ok) raise_error(err, ERRBIT_NUMERIC);
  for (int r = 0; r < kD; ++r) {
    for (int c = 0; c < kD; ++c) {
      Hb[g * kD * kD + r * kD + c] = H[(g * kD + r) * N + g * kD + c];
      Lf[g * kD * kD + r * kD + c] = (ok && c <= r) ? (float)L[r * kD + c] : 0.f;
    }
    Linv[g * kD + r] = ok ? (float)(1.0 / L[r * kD + r]) : 0.f;
  }
}

// x = H_gg^-1 b from the factor: L y = b, L^T x = y.
__device__ __forceinline__ void factor_solve(const float* L, const float* inv, const float b[kD],
                                             float x[kD]) {
  float y[kD];
#pragma unroll
  for (int r = 0; r < kD; ++r) {
    float acc = b[r];
#pragma unroll
    for (int m = 0; m < r; ++m) acc = fmaf(-L[r * kD + m], y[m], acc);
    y[r] = acc * inv[r];
  }
#pragma unroll
  for (int r = kD - 1; r >= 0; --r) {
    float acc = y[r];
#pragma unroll
    for (int m = r + 1; m < kD; ++m) acc = fmaf(-L[m * kD + r], x[m], acc);
    x[r] = acc * inv[r];
  }
}

// Vector (i, g) of D and of its operand images.
__device__ __forceinline__ void store_residual(float* D, int64_t N, char* d_hi, char* d_lo,
                                               int64_t nslab, int64_t i, int64_t g,
                                               const float nv[kD]) {
  uint32_t hi[kD], lo[kD];
#pragma unroll
  for (int j = 0; j < kD; ++j) {
    hi[j] = tc::to_tf32(nv[j]);
    lo[j] = tc::to_tf32(nv[j] - __uint_as_float(hi[j]));
  }
  float* d = D + i * N + g * kD;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    *reinterpret_cast<float4*>(d + 4 * q) =
        make_float4(nv[4 * q], nv[4 * q + 1], nv[4 * q + 2], nv[4 * q + 3]);
    const int64_t off = img::img_off(i, g * kD + 4 * q, nslab);
    *reinterpret_cast<uint4*>(d_hi + off) =
        make_uint4(hi[4 * q], hi[4 * q + 1], hi[4 * q + 2], hi[4 * q + 3]);
    *reinterpret_cast<uint4*>(d_lo + off) =
        make_uint4(lo[4 * q], lo[4 * q + 1], lo[4 * q + 2], lo[4 * q + 3]);
  }
}

// The group steps g = g0 .. g1 - 1 of one block for up to kCplRows rows per CTA. What a step needs from
// global memory is loaded before the steps, all at once: the rows' slice of B^T, their targets
// without codebook `which` (fp32 pairs), their codes, the codebook when it has at most 256 codewords.
// Per group:
//  1. shifted targets, a thread per row: t' = t + H_gg^-1 b_g, t = D_g + C[code_g], b_g = the row's
//     columns of B^T (the block's earlier changes included) - H_gg D_g, the solve a forward and a back
//     substitution in fp32 with the group's factor;
//  2. scores, a thread per codeword (chunks of 256): the fp32 lower bound low_k = s_k - Et_k of every
//     row (8 FMAs) to shared memory; then the two smallest by eight lanes per row (two warp-wide
//     integer reductions per row and warp instead took twice the instructions);
//  3. certificate low_2nd - low_j > 2 Et_j; rows without it are decided exactly, a warp per row: every
//     codeword with low_k <= low_j + 2 Et_j in fp32 pairs, smallest (err, index);
//  4. the new code, D_g, and its change dD_g H[g, g'] added to the later columns, a thread per column.
// Bound: latency of the serial group steps (a 4096 x 4096 sweep has 512 of them, eight warps per SM).
// 4096 x 4096, 256 codewords, one sweep with both losses: 40.2 ms with a kernel per step and group, 13.3
// ms with the steps in this kernel, 7.9 ms with the block products and the losses from operand
// images; loading what the steps need up front, and E's entries ahead in the loss: 5.4 ms; the
// scores' minima from shared memory: 4.7 ms.
constexpr int kCplRows = 32;
constexpr int kCplThreads = 256;
constexpr int kCplPad = kBlockCols + 1;  // row stride of the B^T slice in shared memory

constexpr int kCplScores = kCplThreads + 8;  // row stride of the scores: four rows on distinct banks

struct CplArgs {
  const float* W;      // M x N
  float* D;            // M x N
  const float* H;      // N x N
  const float* Hb;     // [G_cov][8][8]
  const float* Lf;     // [G_cov][8][8]
  const float* Linv;   // [G_cov][8]
  const float* P;      // B^T as [chunks][(g1 - g0) * 8][M]: the chunks' sum, in order
  int chunks;
  char *d_hi, *d_lo;   // the operand images of D, kept up to date
  int64_t nslab;
  int64_t M, N;
  int64_t g0, g1;
  int rows;            // rows per CTA, at most kCplRows
  int which;
  CbList cbs;
};

struct CplShared {
  float B[kCplRows * kCplPad];               // [row][column of the block]
  float2 R[kBlockG][kCplRows][kD];           // targets without `which`: (hi, lo)
  float C[kCplThreads * kD];                 // the codebook (K <= 256)
  int32_t code[kBlockG][kCplRows];
  float S[kCplRows][kCplScores];             // the rows' scores
  float2 nal[kCplThreads];                   // the codewords' (Na, L1)
  float H[2][kD * kD], L[2][kD * kD], inv[2][kD];  // the group's and the next one's
  float T[kCplRows][kD];                     // t'
  float Q[kCplRows][kD];                     // -2 H t'
  float beta[kCplRows];                      // -2 u C Pmax
  float DD[kCplRows][kD];                    // D_g, then its change
  float thr[kCplRows];
  int open[kCplRows];
  int n_open;
};
constexpr size_t kCplSmem = sizeof(CplShared) + 16;

__global__ void __launch_bounds__(kCplThreads)
coupled_block_kernel(const __grid_constant__ CplArgs a, unsigned* err) {
  extern __shared__ __align__(16) char cpl_raw[];
  CplShared& s = *reinterpret_cast<CplShared*>(cpl_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t i0 = (int64_t)blockIdx.x * a.rows;
  const int nr = (int)min((int64_t)a.rows, a.M - i0);
  const int ng = (int)(a.g1 - a.g0), ncol = ng * kD;
  const CbView cw = a.cbs.cb[a.which];
  const SetView wset{a.W, a.N, a.M, a.N / kD, nullptr};
  const float cmul = bound_mult(0);
  const int row8 = tid >> 3, j8 = tid & 7;  // (row, component) threads
  const bool resident = cw.K <= kCplThreads;
  const float* C = resident ? s.C : cw.C;
  for (int e = tid; e < nr * ncol; e += kCplThreads) {
    const int c = e / nr, r = e - c * nr;
    float v = 0.f;
    for (int q = 0; q < a.chunks; ++q) v += __ldg(a.P + ((int64_t)q * ncol + c) * a.M + i0 + r);
    s.B[r * kCplPad + c] = v;
  }
  for (int e = tid; e < nr * ng; e += kCplThreads) {
    const int r = e / ng, gl = e - r * ng;
    float rh[kD], rl[kD];
    others_target(wset, a.cbs, a.which, i0 + r, a.g0 + gl, rh, rl, err);
#pragma unroll
    for (int j = 0; j < kD; ++j) s.R[gl][r][j] = make_float2(rh[j], rl[j]);
    s.code[gl][r] = cw.codes[(i0 + r) * cw.ld + a.g0 + gl];
  }
  if (resident)
    for (int e = tid; e < cw.K * kD; e += kCplThreads) s.C[e] = __ldg(cw.C + e);
  auto load_group = [&](int64_t g, int buf) {  // the group's H block and factor
    if (tid < kD * kD) {
      s.H[buf][tid] = a.Hb[g * kD * kD + tid];
    } else if (tid < 2 * kD * kD) {
      s.L[buf][tid - kD * kD] = a.Lf[g * kD * kD + tid - kD * kD];
    } else if (tid < 2 * kD * kD + kD) {
      s.inv[buf][tid - 2 * kD * kD] = a.Linv[g * kD + tid - 2 * kD * kD];
    }
  };
  load_group(a.g0, 0);
  if (tid == 0) s.n_open = 0;
  __syncthreads();
  for (int64_t g = a.g0; g < a.g1; ++g) {
    const int gl = (int)(g - a.g0), col0 = gl * kD, buf = gl & 1;
    const float* sH = s.H[buf];
    const float* sL = s.L[buf];
    const float* sInv = s.inv[buf];
    float hcol[kD];  // H[g][this thread's column of the block], used at the step's end
    const int col = tid;
    if (col < ncol)
#pragma unroll
      for (int q = 0; q < kD; ++q) hcol[q] = __ldg(a.H + (g * kD + q) * a.N + a.g0 * kD + col);
    if (g + 1 < a.g1) load_group(g + 1, buf ^ 1);
    const bool factor = sInv[0] != 0.f;  // no factor (reported): the code stays
    // this thread's codeword of the first chunk
    float c[kD], n = 0.f, na = 0.f, l1 = 0.f;
#pragma unroll
    for (int j = 0; j < kD; ++j) c[j] = 0.f;
    if (tid < cw.K) {
      load_vec(C + tid * kD, c);
      codeword_terms(c, sH, n, na, l1);
    }
    // 1. shifted targets
    if (tid < nr) {
      const int32_t k = s.code[gl][tid];
      float dg[kD], ck[kD], b[kD];
#pragma unroll
      for (int j = 0; j < kD; ++j) ck[j] = 0.f;
      if (code_ok(k, cw.K, err)) load_vec(C + (int64_t)k * kD, ck);
#pragma unroll
      for (int j = 0; j < kD; ++j) {
        const float2 r = s.R[gl][tid][j];
        dg[j] = pair_minus(r.x, r.y, ck[j]);
        s.DD[tid][j] = dg[j];
      }
#pragma unroll
      for (int q = 0; q < kD; ++q) {
        float hd = 0.f;
#pragma unroll
        for (int m = 0; m < kD; ++m) hd = fmaf(sH[q * kD + m], dg[m], hd);
        b[q] = s.B[tid * kCplPad + col0 + q] - hd;
      }
      float sv[kD];
      factor_solve(sL, sInv, b, sv);
#pragma unroll
      for (int j = 0; j < kD; ++j) s.T[tid][j] = (dg[j] + ck[j]) + sv[j];
    }
    __syncthreads();
    {  // -2 H t' and Pmax, a thread per component
      float q = 0.f, pa = 0.f;
      if (row8 < nr)
#pragma unroll
        for (int j = 0; j < kD; ++j) {
          q = fmaf(sH[j8 * kD + j], s.T[row8][j], q);
          pa = fmaf(fabsf(sH[j8 * kD + j]), fabsf(s.T[row8][j]), pa);
        }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1)
        pa = fmaxf(pa, __shfl_xor_sync(0xffffffffu, pa, off));
      s.Q[row8][j8] = -2.f * q;
      if (j8 == 0) s.beta[row8] = -2.f * kU * cmul * pa;
    }
    __syncthreads();
    // 2. scores, 256 codewords at a time; lane j8 of a row takes every eighth
    float f1 = INFINITY, f2 = INFINITY, e2 = INFINITY;  // smallest, second smallest, 2 Et
    int k1 = 0;
    for (int k0 = 0; k0 < cw.K; k0 += kCplThreads) {
      const int k = k0 + tid, nk = min(kCplThreads, cw.K - k0);
      if (k0 > 0) {
        __syncthreads();  // the earlier chunk's scores have been read
#pragma unroll
        for (int j = 0; j < kD; ++j) c[j] = 0.f;
        n = na = l1 = 0.f;
        if (k < cw.K) {
          load_vec(cw.C + (int64_t)k * kD, c);
          codeword_terms(c, sH, n, na, l1);
        }
      }
      s.nal[tid] = make_float2(na, l1);
      const float nlow = fmaf(-kU * cmul, na, n);
#pragma unroll 4
      for (int r = 0; r < nr; ++r) {
        const float4 q0 = *reinterpret_cast<const float4*>(&s.Q[r][0]);
        const float4 q1 = *reinterpret_cast<const float4*>(&s.Q[r][4]);
        float sc = nlow;
        sc = fmaf(q0.x, c[0], sc);
        sc = fmaf(q0.y, c[1], sc);
        sc = fmaf(q0.z, c[2], sc);
        sc = fmaf(q0.w, c[3], sc);
        sc = fmaf(q1.x, c[4], sc);
        sc = fmaf(q1.y, c[5], sc);
        sc = fmaf(q1.z, c[6], sc);
        sc = fmaf(q1.w, c[7], sc);
        s.S[r][tid] = fmaf(s.beta[r], l1, sc);
      }
      __syncthreads();
      if (row8 < nr) {
        // (a NaN score never wins; it takes f2 down to f1, which opens the row unless a smaller one follows)
#pragma unroll 8
        for (int kk = j8; kk < nk; kk += 8) {
          const float sc = s.S[row8][kk];
          k1 = sc < f1 ? k0 + kk : k1;  // ties: the smaller index
          f2 = fminf(f2, fmaxf(f1, sc));
          f1 = fminf(f1, sc);
        }
        if (k1 >= k0) {
          const float2 t = s.nal[k1 - k0];
          e2 = 2.f * kU * cmul * t.x - 2.f * s.beta[row8] * t.y;
        }
      }
    }
    // 3. the row's smallest over its eight lanes, certificate
    {
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) {
        const float o1 = __shfl_xor_sync(0xffffffffu, f1, off);
        const float o2 = __shfl_xor_sync(0xffffffffu, f2, off);
        const int ok = __shfl_xor_sync(0xffffffffu, k1, off);
        const float oe = __shfl_xor_sync(0xffffffffu, e2, off);
        const bool take = o1 < f1 || (o1 == f1 && ok < k1);
        f2 = fminf(fminf(f2, o2), fmaxf(f1, o1));
        if (take) {
          f1 = o1;
          k1 = ok;
          e2 = oe;
        }
      }
      if (j8 == 0 && row8 < nr && factor) {
        const bool found = f1 < INFINITY;
        if (cw.K == 1 || (found && f2 - f1 > e2)) {
          s.code[gl][row8] = k1;
        } else {
          s.thr[row8] = found ? __fadd_ru(f1, e2) : INFINITY;
          s.open[atomicAdd(&s.n_open, 1)] = row8;
        }
      }
    }
    __syncthreads();
    if (s.n_open > 0) {  // exact decisions, a warp per row
      for (int q = warp; q < s.n_open; q += kCplThreads / 32) {
        const int r = s.open[q];
        const float thr = s.thr[r], nbeta = s.beta[r];
        float t[kD], zero[kD], m2q[kD];
#pragma unroll
        for (int j = 0; j < kD; ++j) {
          t[j] = s.T[r][j];
          zero[j] = 0.f;
          m2q[j] = s.Q[r][j];
        }
        float bh = INFINITY, bl = 0.f;
        int bk = 0x7fffffff;
        for (int k = lane; k < cw.K; k += 32) {
          float cv[kD], kn, kna, kl1;
          load_vec(C + (int64_t)k * kD, cv);
          codeword_terms(cv, sH, kn, kna, kl1);
          if (low_from(kn, kna, kl1, cv, m2q, nbeta, cmul) <= thr) {
            float eh, el;
            dfl::quad_err(t, zero, cv, sH, eh, el);
            if (dfl::less(eh, el, k, bh, bl, bk)) {
              bh = eh;
              bl = el;
              bk = k;
            }
          }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          const float oh = __shfl_xor_sync(0xffffffffu, bh, off);
          const float ol = __shfl_xor_sync(0xffffffffu, bl, off);
          const int ok = __shfl_xor_sync(0xffffffffu, bk, off);
          if (dfl::less(oh, ol, ok, bh, bl, bk)) {
            bh = oh;
            bl = ol;
            bk = ok;
          }
        }
        if (lane == 0) {
          if (bk == 0x7fffffff)
            raise_error(err, ERRBIT_NUMERIC);  // no candidate: non-finite scores (the code stays)
          else
            s.code[gl][r] = bk;
        }
      }
      __syncthreads();
      if (tid == 0) s.n_open = 0;
    }
    // 4. the decision: code, D_g and its operand images, the change of D_g
    if (tid < nr) {
      const int64_t i = i0 + tid;
      const int32_t kn = s.code[gl][tid];
      if (factor && code_ok(kn, cw.K, err)) {
        cw.codes[i * cw.ld + g] = kn;
        float ck[kD], nv[kD];
        load_vec(C + (int64_t)kn * kD, ck);
#pragma unroll
        for (int j = 0; j < kD; ++j) {
          const float2 r = s.R[gl][tid][j];
          nv[j] = pair_minus(r.x, r.y, ck[j]);
          s.DD[tid][j] = nv[j] - s.DD[tid][j];
        }
        store_residual(a.D, a.N, a.d_hi, a.d_lo, a.nslab, i, g, nv);
      } else {
#pragma unroll
        for (int j = 0; j < kD; ++j) s.DD[tid][j] = 0.f;
      }
    }
    __syncthreads();
    if (col >= col0 + kD && col < ncol) {
#pragma unroll 4
      for (int r = 0; r < nr; ++r) {
        const float4 d0 = *reinterpret_cast<const float4*>(&s.DD[r][0]);
        const float4 d1 = *reinterpret_cast<const float4*>(&s.DD[r][4]);
        float acc = s.B[r * kCplPad + col];
        acc = fmaf(d0.x, hcol[0], acc);
        acc = fmaf(d0.y, hcol[1], acc);
        acc = fmaf(d0.z, hcol[2], acc);
        acc = fmaf(d0.w, hcol[3], acc);
        acc = fmaf(d1.x, hcol[4], acc);
        acc = fmaf(d1.y, hcol[5], acc);
        acc = fmaf(d1.z, hcol[6], acc);
        acc = fmaf(d1.w, hcol[7], acc);
        s.B[r * kCplPad + col] = acc;
      }
    }
    __syncthreads();
  }
}

// ---- the same step in three parts, for the tensor-core arg-min; B^T summed over the chunks first.

// P[0] += P[1] + ... in order (n elements each).
__global__ void __launch_bounds__(256)
coupled_sum_chunks_kernel(float* __restrict__ P, int chunks, int64_t n) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    float v = P[e];
    for (int q = 1; q < chunks; ++q) v += P[q * n + e];
    P[e] = v;
  }
}

// Shifted targets of group g (step 1 of coupled_block_kernel), a thread per row: Tp[i][8].
__global__ void __launch_bounds__(128)
coupled_target_kernel(const __grid_constant__ CplArgs a, int64_t g, const float* __restrict__ Bt,
                      float* __restrict__ Tp, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  __shared__ float sH[kD * kD], sL[kD * kD], sInv[kD];
  if (threadIdx.x < kD * kD) {
    sH[threadIdx.x] = a.Hb[g * kD * kD + threadIdx.x];
    sL[threadIdx.x] = a.Lf[g * kD * kD + threadIdx.x];
  }
  if (threadIdx.x < kD) sInv[threadIdx.x] = a.Linv[g * kD + threadIdx.x];
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.M) return;
  const CbView cw = a.cbs.cb[a.which];
  const int col0 = (int)(g - a.g0) * kD;
  float dg[kD], ck[kD], b[kD], sv[kD];
  load_vec(a.D + i * a.N + g * kD, dg);
#pragma unroll
  for (int j = 0; j < kD; ++j) ck[j] = 0.f;
  const int32_t k = cw.codes[i * cw.ld + g];
  if (code_ok(k, cw.K, err)) load_vec(cw.C + (int64_t)k * kD, ck);
#pragma unroll
  for (int q = 0; q < kD; ++q) {
    float hd = 0.f;
#pragma unroll
    for (int m = 0; m < kD; ++m) hd = fmaf(sH[q * kD + m], dg[m], hd);
    b[q] = Bt[(int64_t)(col0 + q) * a.M + i] - hd;
  }
  factor_solve(sL, sInv, b, sv);  // (no factor: zeros)
#pragma unroll
  for (int j = 0; j < kD; ++j) sv[j] = (dg[j] + ck[j]) + sv[j];
  float* t = Tp + i * kD;
  *reinterpret_cast<float4*>(t) = make_float4(sv[0], sv[1], sv[2], sv[3]);
  *reinterpret_cast<float4*>(t + 4) = make_float4(sv[4], sv[5], sv[6], sv[7]);
}

// Applies the decisions of group g (step 4 of coupled_block_kernel): 32 rows per CTA, a lane each; the
// first warp takes the code, D_g and its change, all eight the later columns of the block in turn.
__global__ void __launch_bounds__(256)
coupled_apply_kernel(const __grid_constant__ CplArgs a, int64_t g, const int32_t* __restrict__ code,
                     float* __restrict__ Bt, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  __shared__ float sDD[kD][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * 32 + lane;
  const CbView cw = a.cbs.cb[a.which];
  if (a.Linv[g * kD] == 0.f) return;  // no factor (reported): the codes stay
  if (warp == 0) {
    float dd[kD];
#pragma unroll
    for (int j = 0; j < kD; ++j) dd[j] = 0.f;
    if (i < a.M) {
      const int32_t kn = code[i];
      if (code_ok(kn, cw.K, err)) {
        cw.codes[i * cw.ld + g] = kn;
        const SetView wset{a.W, a.N, a.M, a.N / kD, nullptr};
        float rh[kD], rl[kD], ck[kD], nv[kD];
        others_target(wset, a.cbs, a.which, i, g, rh, rl, err);
        load_vec(cw.C + (int64_t)kn * kD, ck);
        load_vec(a.D + i * a.N + g * kD, dd);
#pragma unroll
        for (int j = 0; j < kD; ++j) {
          nv[j] = pair_minus(rh[j], rl[j], ck[j]);
          dd[j] = nv[j] - dd[j];
        }
        store_residual(a.D, a.N, a.d_hi, a.d_lo, a.nslab, i, g, nv);
      }
    }
#pragma unroll
    for (int j = 0; j < kD; ++j) sDD[j][lane] = dd[j];
  }
  __syncthreads();
  if (i >= a.M) return;
  float dd[kD];
#pragma unroll
  for (int j = 0; j < kD; ++j) dd[j] = sDD[j][lane];
  const int ncol = (int)(a.g1 - a.g0) * kD;
#pragma unroll 4
  for (int col = (int)(g + 1 - a.g0) * kD + warp; col < ncol; col += 8) {
    float acc = Bt[(int64_t)col * a.M + i];
#pragma unroll
    for (int q = 0; q < kD; ++q)
      acc = fmaf(dd[q], __ldg(a.H + (g * kD + q) * a.N + a.g0 * kD + col), acc);
    Bt[(int64_t)col * a.M + i] = acc;
  }
}

// *out = sum of part[0 .. n) (one CTA, strided sums and a tree: a fixed order).
__global__ void __launch_bounds__(1024)
sum_parts_kernel(const double* __restrict__ part, int64_t n, double* out) {
  __shared__ double red[1024];
  double s = 0.0;
  for (int64_t q = threadIdx.x; q < n; q += blockDim.x) s += part[q];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

// Whether a sweep's steps go through the tensor-core arg-min. coupled_block_kernel takes about 10 ns per
// codeword and step (more above 16384 codewords, whose open rows are long scans) for each wave of blocks;
// the arg-min takes about 30 us per step in its five launches, 4 ns more per codeword, and next to
// nothing per row. Block kernel / arg-min, one sweep with both losses: 4096 x 1024, 4096 codewords 6.4 / 6.9
// ms, 8192 13.2 / 10.9, 65536 142 / 64; 6000 x 1024 (two waves), 1024 codewords 3.6 / 4.2, 2048 6.2 / 5.4;
// 9800 x 512 (three), 256 1.3 / 1.8, 1024 2.5 / 2.1; 16384 x 512 (four), 256 1.7 / 1.9, 600 2.7 / 2.2;
// 28672 x 512 (six), 256 2.6 / 2.6, 4096 16 / 5.
bool coupled_by_argmin(int64_t M, int K, int rows, int nsm) {
  const int64_t waves = ceil_div(ceil_div(M, rows), nsm);
  return K * waves * waves > 6000;
}

}  // namespace

crvq_status launch_coupled_sweep(const float* W, int64_t M, int64_t N, const float* H,
                                 const CbList& cbs_in, int which, int sweeps, double* loss_dev,
                                 cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  const int nsm = sm_count();
  CbList cbs = cbs_in;
  const CbView cw = cbs.cb[which];
  const int64_t G_cov = cw.G_cov;
  const int64_t chunks = img_k_chunks(N);
  const int64_t n_part = ceil_div(M, (int64_t)128) * ceil_div(N, (int64_t)256);
  const size_t h_img = img_bytes(N, N), d_img = img_bytes(M, N);
  Scratch mD, mI, mB, mP, mF;
  CRVQ_TRY(mD.alloc((size_t)M * N * sizeof(float), stream));
  CRVQ_TRY(mI.alloc(2 * (h_img + d_img), stream));
  CRVQ_TRY(mB.alloc((size_t)chunks * kBlockCols * M * sizeof(float), stream));
  CRVQ_TRY(mP.alloc((size_t)n_part * sizeof(double), stream));
  CRVQ_TRY(mF.alloc((size_t)std::max<int64_t>(G_cov, 1) * (2 * kD * kD + kD) * sizeof(float),
                    stream));
  float* D = mD.as<float>();
  char* h_hi = mI.as<char>();
  char* h_lo = h_hi + h_img;
  char* d_hi = h_lo + h_img;
  char* d_lo = d_hi + d_img;
  float* Hb = mF.as<float>();
  float* Lf = Hb + G_cov * kD * kD;
  float* Linv = Lf + G_cov * kD * kD;
  {
    ProfScope ps("coupled_residual", stream, (double)M * N * 8.0);
    residual_kernel<<<(unsigned)std::min<int64_t>(ceil_div(M * (N / kD), 256), 16 * nsm), 256, 0,
                      stream>>>(W, M, N, cbs, which, D, err);
    CRVQ_LAUNCHED();
    block_factor_kernel<<<(unsigned)ceil_div(std::max<int64_t>(G_cov, 1), 128), 128, 0,
                          stream>>>(H, N, G_cov, Hb, Lf, Linv, err);
    CRVQ_LAUNCHED();
  }
  // operand images of H and D; the sweep keeps D's up to date
  CRVQ_TRY(launch_images(H, nullptr, nullptr, N, N, h_hi, h_lo, stream));
  CRVQ_TRY(launch_images(D, nullptr, nullptr, M, N, d_hi, d_lo, stream));
  auto loss_into = [&](double* out) -> crvq_status {  // tr(D H D^T) = sum (D H) . D
    CRVQ_TRY(launch_img_dot(d_hi, d_lo, M, h_hi, h_lo, N, N, D, mP.as<double>(), stream));
    sum_parts_kernel<<<1, 1024, 0, stream>>>(mP.as<double>(), n_part, out);
    CRVQ_LAUNCHED();
    return CRVQ_OK;
  };
  if (loss_dev) CRVQ_TRY(loss_into(loss_dev));
  // rows per CTA: every SM gets rows, at least eight of them (a group step is mostly latency)
  const int rows = (int)std::min<int64_t>(kCplRows, std::max<int64_t>(8, ceil_div(M, nsm)));
  const bool by_argmin = coupled_by_argmin(M, cw.K, rows, nsm);
  Scratch mT, mW;
  EncodeExtras ex;
  if (by_argmin) {
    CRVQ_TRY(mT.alloc((size_t)M * (kD + 1) * sizeof(float), stream));
    const size_t wbytes = argmin_scratch_bytes(M, 1, cw.K);
    CRVQ_TRY(mW.alloc(wbytes, stream));
    ex.work = mW.as<char>();
    ex.work_bytes = wbytes;
  }
  for (int sw = 0; sw < sweeps; ++sw) {
    for (int64_t b0 = 0; b0 < G_cov; b0 += kBlockG) {
      const int64_t b1 = std::min<int64_t>(G_cov, b0 + kBlockG);
      const int nc = (int)((b1 - b0) * kD);
      // B^T for the block's channels, with every decision so far in D
      CRVQ_TRY(launch_img_gemm_chunks(h_hi, h_lo, b0 * kD, nc, d_hi, d_lo, M, N, mB.as<float>(),
                                      stream));
      const CplArgs ca{W, D, H, Hb, Lf, Linv, mB.as<float>(), (int)chunks, d_hi, d_lo,
                       ceil_div(N, (int64_t)img::kSlabK), M, N, b0, b1, rows, which, cbs};
      ProfScope ps("coupled_block", stream, (double)M * (b1 - b0) * cw.K);
      if (!by_argmin) {
        CRVQ_TRY(smem_limit((const void*)coupled_block_kernel, kCplSmem));
        coupled_block_kernel<<<(unsigned)ceil_div(M, rows), kCplThreads, kCplSmem, stream>>>(ca, err);
        CRVQ_LAUNCHED();
        continue;
      }
      float* Bt = mB.as<float>();
      float* Tp = mT.as<float>();
      int32_t* code = reinterpret_cast<int32_t*>(Tp + M * kD);
      if (chunks > 1) {
        const int64_t n = (int64_t)nc * M;
        CRVQ_CUDA(launch_pdl(coupled_sum_chunks_kernel, dim3((unsigned)std::min<int64_t>(
                             ceil_div(n, 256), 16 * nsm)), dim3(256), 0, stream, Bt, (int)chunks, n));
        CRVQ_LAUNCHED();
      }
      CbList one{};
      one.n = 1;
      one.cb[0] = CbView{cw.C, code, 1, 1, cw.K};
      for (int64_t g = b0; g < b1; ++g) {
        CRVQ_CUDA(launch_pdl(coupled_target_kernel, dim3((unsigned)ceil_div(M, (int64_t)128)),
                             dim3(128), 0, stream, ca, g, Bt, Tp, err));
        CRVQ_LAUNCHED();
        CRVQ_TRY(launch_encode_beam(SetView{Tp, kD, M, 1, Hb + g * kD * kD}, one, 0, 1, false,
                                    nullptr, ex, stream));
        CRVQ_CUDA(launch_pdl(coupled_apply_kernel, dim3((unsigned)ceil_div(M, (int64_t)32)), dim3(256),
                             0, stream, ca, g, code, Bt, err));
        CRVQ_LAUNCHED();
      }
    }
    if (loss_dev) CRVQ_TRY(loss_into(loss_dev + 1 + sw));
  }
  return CRVQ_OK;
}

}  // namespace crvq
