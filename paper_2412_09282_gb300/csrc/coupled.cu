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
// decisions, update) and the round trips of B^T through L2 are gone.
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

// D = W - sum over the covering codebooks of C[code] (fp32 pairs, rounded once), M x N.
__global__ void __launch_bounds__(256)
residual_kernel(const float* __restrict__ W, int64_t M, int64_t N, CbList cbs,
                float* __restrict__ D, unsigned* err) {
  const int64_t G = N / kD;
  const SetView set{W, N, M, G, nullptr};
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < M * G;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = v / G, g = v % G;
    float rh[kD], rl[kD];
    dfl::target(set, cbs, cbs.n, i, g, rh, rl, err);
    float* o = D + i * N + g * kD;
    *reinterpret_cast<float4*>(o) = make_float4(__fadd_rn(rh[0], rl[0]), __fadd_rn(rh[1], rl[1]),
                                                __fadd_rn(rh[2], rl[2]), __fadd_rn(rh[3], rl[3]));
    *reinterpret_cast<float4*>(o + 4) =
        make_float4(__fadd_rn(rh[4], rl[4]), __fadd_rn(rh[5], rl[5]), __fadd_rn(rh[6], rl[6]),
                    __fadd_rn(rh[7], rl[7]));
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

// The group steps g = g0 .. g1 - 1 of one block for up to kCplRows rows per CTA. Per group:
//  1. shifted targets, a thread per row: t' = t + H_gg^-1 b_g, t = D_g + C[code_g], b_g = the row's
//     columns of B^T (shared memory, the block's earlier changes included) - H_gg D_g, the solve a
//     forward and a back substitution in fp32 with the group's factor;
//  2. scores, a thread per codeword (chunks of 256): the fp32 lower bound low_k = s_k - Et_k of every
//     row (8 FMAs), the two smallest of a warp's 32 by integer minima over order-preserving keys
//     (redux), the two smallest of all by the row's eight lanes;
//  3. certificate low_2nd - low_j > 2 Et_j; rows without it are decided exactly, a warp per row: every
//     codeword with low_k <= low_j + 2 Et_j in fp32 pairs, smallest (err, index);
//  4. the new code, D_g from W, and its change dD_g H[g, g'] added to the later columns, a thread per
//     column.
// Bound: latency of the serial group steps (six barriers and about 3 k cycles each at 32 rows).
// 4096 x 4096, 256 codewords, one sweep with both losses: 40.2 ms with a kernel per step and group, 13.3
// ms with this one.
constexpr int kCplRows = 32;
constexpr int kCplThreads = 256;
constexpr int kCplPad = kBlockCols + 1;  // row stride of the B^T slice in shared memory

// Order-preserving map of fp32 to uint32 (NaN above every number).
__device__ __forceinline__ uint32_t order_key(float x) {
  const uint32_t b = __float_as_uint(x);
  return x != x ? 0xffffffffu : ((b >> 31) ? ~b : b | 0x80000000u);
}
__device__ __forceinline__ float order_val(uint32_t k) {
  return __uint_as_float((k >> 31) ? k & 0x7fffffffu : ~k);
}

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

__global__ void __launch_bounds__(kCplThreads)
coupled_block_kernel(const __grid_constant__ CplArgs a, unsigned* err) {
  __shared__ float sB[kCplRows * kCplPad];            // [row][column of the block]
  __shared__ __align__(16) float sH[kD * kD];
  __shared__ float sL[kD * kD], sInv[kD];
  __shared__ __align__(16) float sT[kCplRows][kD];    // t'
  __shared__ __align__(16) float sQ[kCplRows][kD];    // -2 H t'
  __shared__ float sPmax[kCplRows];
  __shared__ __align__(16) float sDD[kCplRows][kD];   // change of D_g
  __shared__ uint32_t sV1[kCplRows][8], sV2[kCplRows][8];  // per warp: smallest, second smallest key
  __shared__ int sK1[kCplRows][8];
  __shared__ float sE1[kCplRows][8];                  // 2 Et of the smallest
  __shared__ int sCode[kCplRows];
  __shared__ float sThr[kCplRows];
  __shared__ int sOpen[kCplRows];
  __shared__ int n_open;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t i0 = (int64_t)blockIdx.x * a.rows;
  const int nr = (int)min((int64_t)a.rows, a.M - i0);
  const int ncol = (int)(a.g1 - a.g0) * kD;
  const CbView cw = a.cbs.cb[a.which];
  const SetView wset{a.W, a.N, a.M, a.N / kD, nullptr};
  const float cmul = bound_mult(0);
  const int row8 = tid >> 3, j8 = tid & 7;  // (row, component) threads
  for (int e = tid; e < nr * ncol; e += kCplThreads) {
    const int c = e / nr, r = e - c * nr;
    float s = 0.f;
    for (int q = 0; q < a.chunks; ++q) s += __ldg(a.P + ((int64_t)q * ncol + c) * a.M + i0 + r);
    sB[r * kCplPad + c] = s;
  }
  for (int64_t g = a.g0; g < a.g1; ++g) {
    const int col0 = (int)(g - a.g0) * kD;
    // loads that do not depend on the previous group's decision
    float hcol[kD];  // H[g][this thread's column of the block]
    const int col = tid;
    if (col < ncol)
#pragma unroll
      for (int q = 0; q < kD; ++q) hcol[q] = __ldg(a.H + (g * kD + q) * a.N + a.g0 * kD + col);
    float dold = 0.f;
    if (row8 < nr) dold = a.D[(i0 + row8) * a.N + g * kD + j8];
    if (tid < kD * kD) {
      sH[tid] = a.Hb[g * kD * kD + tid];
      sL[tid] = a.Lf[g * kD * kD + tid];
    }
    if (tid < kD) sInv[tid] = a.Linv[g * kD + tid];
    if (tid == 0) n_open = 0;
    if (row8 < nr) sDD[row8][j8] = dold;  // D_g until the decision
    __syncthreads();  // (and the previous group's changes of sB are visible)
    const bool factor = sInv[0] != 0.f;  // no factor (reported): the code stays
    // 1. shifted targets
    if (tid < nr) {
      const int64_t i = i0 + tid;
      float dg[kD], b[kD];
#pragma unroll
      for (int j = 0; j < kD; ++j) dg[j] = sDD[tid][j];
#pragma unroll
      for (int q = 0; q < kD; ++q) {
        float hd = 0.f;
#pragma unroll
        for (int c = 0; c < kD; ++c) hd = fmaf(sH[q * kD + c], dg[c], hd);
        b[q] = sB[tid * kCplPad + col0 + q] - hd;
      }
      // H_gg s = b: L y = b, L^T s = y
      float y[kD], sv[kD];
#pragma unroll
      for (int r = 0; r < kD; ++r) {
        float acc = b[r];
#pragma unroll
        for (int m = 0; m < r; ++m) acc = fmaf(-sL[r * kD + m], y[m], acc);
        y[r] = acc * sInv[r];
      }
#pragma unroll
      for (int r = kD - 1; r >= 0; --r) {
        float acc = y[r];
#pragma unroll
        for (int m = r + 1; m < kD; ++m) acc = fmaf(-sL[m * kD + r], sv[m], acc);
        sv[r] = acc * sInv[r];
      }
      const int32_t k = cw.codes[i * cw.ld + g];
      const bool kok = code_ok(k, cw.K, err);
      float c[kD];
#pragma unroll
      for (int j = 0; j < kD; ++j) c[j] = 0.f;
      if (kok) load_vec(cw.C + (int64_t)k * kD, c);
#pragma unroll
      for (int j = 0; j < kD; ++j) sT[tid][j] = (dg[j] + c[j]) + sv[j];
      sCode[tid] = k;
    }
    __syncthreads();
    if (row8 < kCplRows) {  // -2 H t' and Pmax, a thread per component
      float q = 0.f, pa = 0.f;
      if (row8 < nr)
#pragma unroll
        for (int j = 0; j < kD; ++j) {
          q = fmaf(sH[j8 * kD + j], sT[row8][j], q);
          pa = fmaf(fabsf(sH[j8 * kD + j]), fabsf(sT[row8][j]), pa);
        }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1)
        pa = fmaxf(pa, __shfl_xor_sync(0xffffffffu, pa, off));
      sQ[row8][j8] = -2.f * q;
      if (j8 == 0) sPmax[row8] = pa;
    }
    __syncthreads();
    // 2. scores, 256 codewords at a time; each warp keeps its two smallest per row
    for (int k0 = 0; k0 < cw.K; k0 += kCplThreads) {
      const int k = k0 + tid;
      float c[kD], n = 0.f, na = 0.f, l1 = 0.f;
#pragma unroll
      for (int j = 0; j < kD; ++j) c[j] = 0.f;
      if (k < cw.K) {
        load_vec(cw.C + (int64_t)k * kD, c);
        codeword_terms(c, sH, n, na, l1);
      }
      const float nlow = fmaf(-kU * cmul, na, n);
#pragma unroll 4
      for (int r = 0; r < nr; ++r) {
        const float4 q0 = *reinterpret_cast<const float4*>(&sQ[r][0]);
        const float4 q1 = *reinterpret_cast<const float4*>(&sQ[r][4]);
        const float pmax = sPmax[r];
        float sc = nlow;
        sc = fmaf(q0.x, c[0], sc);
        sc = fmaf(q0.y, c[1], sc);
        sc = fmaf(q0.z, c[2], sc);
        sc = fmaf(q0.w, c[3], sc);
        sc = fmaf(q1.x, c[4], sc);
        sc = fmaf(q1.y, c[5], sc);
        sc = fmaf(q1.z, c[6], sc);
        sc = fmaf(q1.w, c[7], sc);
        sc = fmaf(-2.f * kU * cmul * pmax, l1, sc);
        const uint32_t key = k < cw.K ? order_key(sc) : 0xffffffffu;
        const uint32_t m1 = __reduce_min_sync(0xffffffffu, key);
        const int src = __ffs(__ballot_sync(0xffffffffu, key == m1)) - 1;
        const uint32_t m2 = __reduce_min_sync(0xffffffffu, lane == src ? 0xffffffffu : key);
        if (lane == src) {
          const float e2 = 2.f * kU * cmul * (na + 2.f * pmax * l1);
          if (k0 == 0) {
            sV1[r][warp] = m1;
            sV2[r][warp] = m2;
            sK1[r][warp] = k;
            sE1[r][warp] = e2;
          } else {  // (the warp's earlier chunks; strictly below: ties keep the smaller index)
            const uint32_t v1 = sV1[r][warp];
            if (m1 < v1) {
              sV2[r][warp] = min(v1, m2);
              sV1[r][warp] = m1;
              sK1[r][warp] = k;
              sE1[r][warp] = e2;
            } else {
              sV2[r][warp] = min(sV2[r][warp], m1);
            }
          }
        }
      }
      __syncwarp();
    }
    __syncthreads();
    // 3. the row's smallest over its eight lanes (warps' entries), certificate
    if (row8 < kCplRows) {
      uint32_t v1 = 0xffffffffu, v2 = 0xffffffffu;
      int k1 = 0;
      float e2 = 0.f;
      if (row8 < nr) {
        v1 = sV1[row8][j8];
        v2 = sV2[row8][j8];
        k1 = sK1[row8][j8];
        e2 = sE1[row8][j8];
      }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) {
        const uint32_t o1 = __shfl_xor_sync(0xffffffffu, v1, off);
        const uint32_t o2 = __shfl_xor_sync(0xffffffffu, v2, off);
        const int ok = __shfl_xor_sync(0xffffffffu, k1, off);
        const float oe = __shfl_xor_sync(0xffffffffu, e2, off);
        const bool take = o1 < v1 || (o1 == v1 && ok < k1);
        v2 = min(min(v2, o2), max(v1, o1));
        if (take) {
          v1 = o1;
          k1 = ok;
          e2 = oe;
        }
      }
      if (j8 == 0 && row8 < nr && factor) {
        const float low1 = order_val(v1);
        const bool cert = cw.K == 1 || (v1 != 0xffffffffu && order_val(v2) - low1 > e2) ||
                          (v1 != 0xffffffffu && v2 == 0xffffffffu && isfinite(e2));
        if (cert) {
          sCode[row8] = k1;
        } else {
          sThr[row8] = v1 != 0xffffffffu ? __fadd_ru(low1, e2) : INFINITY;
          sOpen[atomicAdd(&n_open, 1)] = row8;
        }
      }
    }
    __syncthreads();
    for (int q = warp; q < n_open; q += kCplThreads / 32) {  // exact decisions, a warp per row
      const int r = sOpen[q];
      const float thr = sThr[r];
      float t[kD], zero[kD], m2q[kD];
#pragma unroll
      for (int j = 0; j < kD; ++j) {
        t[j] = sT[r][j];
        zero[j] = 0.f;
        m2q[j] = sQ[r][j];
      }
      const float nbeta = -2.f * kU * cmul * sPmax[r];
      float bh = INFINITY, bl = 0.f;
      int bk = 0x7fffffff;
      for (int k = lane; k < cw.K; k += 32) {
        float c[kD], n, na, l1;
        load_vec(cw.C + (int64_t)k * kD, c);
        codeword_terms(c, sH, n, na, l1);
        if (low_from(n, na, l1, c, m2q, nbeta, cmul) <= thr) {
          float eh, el;
          dfl::quad_err(t, zero, c, sH, eh, el);
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
          sCode[r] = bk;
      }
    }
    __syncthreads();
    // 4. the decision: code, D_g from W, the change of D_g
    if (tid < nr && factor) {
      const int64_t i = i0 + tid;
      const int32_t kn = sCode[tid];
      if (code_ok(kn, cw.K, err)) {
        cw.codes[i * cw.ld + g] = kn;
        float rh[kD], rl[kD];
        dfl::target(wset, a.cbs, a.cbs.n, i, g, rh, rl, err);  // (reads the code just written)
        float* d = a.D + i * a.N + g * kD;
        uint32_t hi[kD], lo[kD];
#pragma unroll
        for (int j = 0; j < kD; ++j) {
          const float nv = __fadd_rn(rh[j], rl[j]);
          d[j] = nv;
          sDD[tid][j] = nv - sDD[tid][j];
          hi[j] = tc::to_tf32(nv);
          lo[j] = tc::to_tf32(nv - __uint_as_float(hi[j]));
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int64_t off = img::img_off(i, g * kD + 4 * q, a.nslab);
          *reinterpret_cast<uint4*>(a.d_hi + off) =
              make_uint4(hi[4 * q], hi[4 * q + 1], hi[4 * q + 2], hi[4 * q + 3]);
          *reinterpret_cast<uint4*>(a.d_lo + off) =
              make_uint4(lo[4 * q], lo[4 * q + 1], lo[4 * q + 2], lo[4 * q + 3]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < kD; ++j) sDD[tid][j] = 0.f;
      }
    }
    __syncthreads();
    if (factor && col >= col0 + kD && col < ncol) {
#pragma unroll 4
      for (int r = 0; r < nr; ++r) {
        const float4 d0 = *reinterpret_cast<const float4*>(&sDD[r][0]);
        const float4 d1 = *reinterpret_cast<const float4*>(&sDD[r][4]);
        float acc = sB[r * kCplPad + col];
        acc = fmaf(d0.x, hcol[0], acc);
        acc = fmaf(d0.y, hcol[1], acc);
        acc = fmaf(d0.z, hcol[2], acc);
        acc = fmaf(d0.w, hcol[3], acc);
        acc = fmaf(d1.x, hcol[4], acc);
        acc = fmaf(d1.y, hcol[5], acc);
        acc = fmaf(d1.z, hcol[6], acc);
        acc = fmaf(d1.w, hcol[7], acc);
        sB[r * kCplPad + col] = acc;
      }
    }
    __syncthreads();
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
                      stream>>>(W, M, N, cbs, D, err);
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
      coupled_block_kernel<<<(unsigned)ceil_div(M, rows), kCplThreads, 0, stream>>>(ca, err);
      CRVQ_LAUNCHED();
    }
    if (loss_dev) CRVQ_TRY(loss_into(loss_dev + 1 + sw));
  }
  return CRVQ_OK;
}

}  // namespace crvq
