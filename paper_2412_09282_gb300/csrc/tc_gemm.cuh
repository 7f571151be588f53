// The d x d diagonal blocks of X^T X (App. A.2) on the tensor cores (tcgen05, sm_103a), fp32-accurate
// via the 3xTF32 split, with the accumulator in tensor memory.
//
// Each fp32 operand x is split into x_hi = tf32(x) and x_lo = tf32(x - x_hi); the product
// uses a_hi b_hi + a_hi b_lo + a_lo b_hi (the dropped a_lo b_lo term and the rounding of the
// lo parts are ~2^-22 relative), accumulated in fp32 by the tensor core.
//
// K is staged 16 at a time through four shared-memory stages, each filled by its own 128 threads (a
// thread per row: load ahead in registers, split, store) while the tensor core works on the earlier
// ones; one more warp issues the MMAs in K order. Operands sit in shared memory in the canonical
// K-major layout without swizzle: 8-row x 16-byte core matrices, consecutive along K (LBO = 128 B), 8-row
// groups SBO = (BK / 4) * 128 B apart. Every wait on an mbarrier is bounded (~2 s of
// %globaltimer); on expiry the kernel records ERRBIT_TIMEOUT, stops issuing and exits
// after freeing its tensor memory. (The dense products run from operand images: tc_gemm.cu.)
#pragma once

#include "common.cuh"
#include "tc_ops.cuh"

namespace crvq {
namespace tc {

constexpr int kBM = 128, kBK = 16;
constexpr int kAStageBytes = kBM * kBK * 4;            // one of hi / lo

// Byte offset of element (r, k) in a K-major no-swizzle tile with kBK columns.
__device__ __forceinline__ uint32_t tile_off(int r, int k) {
  return (uint32_t)(((r >> 3) * (kBK / 4) + (k >> 2)) * 128 + (r & 7) * 16 + (k & 3) * 4);
}

// kBK values of a row from src (null: zeros), n of them valid (zeros past them).
__device__ __forceinline__ void load_row(const float* src, int64_t n, bool aligned, float v[kBK]) {
  if (src && n >= kBK && aligned) {
#pragma unroll
    for (int q = 0; q < kBK / 4; ++q) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(src) + q);
      v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < kBK; ++q) v[q] = src && q < n ? src[q] : 0.f;
  }
}

// Splits the loaded values of row r into tf32 hi / lo and stores both.
__device__ __forceinline__ void split_store(const float v[kBK], int r, char* hi, char* lo) {
#pragma unroll
  for (int q = 0; q < kBK / 4; ++q) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      h[j] = to_tf32(v[4 * q + j]);
      l[j] = to_tf32(v[4 * q + j] - __uint_as_float(h[j]));
    }
    const uint32_t off = tile_off(r, 4 * q);
    *reinterpret_cast<uint4*>(hi + off) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(lo + off) = make_uint4(l[0], l[1], l[2], l[3]);
  }
}

// Diagonal d x d blocks (d = 8) of S = A A^T for the rows of A taken in a given order (the
// Hessian blocks of the original or of the importance-sorted channel groups): one CTA per
// 128-row tile and K chunk. A block only pairs rows of the same tile, so the tile's operand is
// split once and is both MMA operands (M = N = 128, half the shared memory and staging work of
// a 128 x 256 tile). Entry (a, b) of a block is taken as the dense product's tile path takes
// it: the dense S keeps D(A row min(p, q), B row max(p, q)) for stored rows p, q (its upper
// triangle, mirrored), so here too the row with the smaller stored index is the A side. Every
// tcgen05 output element is the same function of its A row, B row and K order wherever it sits
// in a tile, so the blocks equal the dense S's entries bit for bit.
//
// Bound: the serial MMAs of a CTA (1024 tokens: 384 of 128 x 128 x 8, about 17 us at the tf32 rate). With
// 128 threads that filled two stages in turn, two block barriers per 16 tokens, a launch over 1024 tokens
// took 51 us; now 37.
constexpr int kDiagStages = 4;                              // = groups of 128 threads
constexpr int kDiagThreads = kDiagStages * kBM + 32;
constexpr int kDiagStageBytes = 2 * kAStageBytes;           // hi + lo, 16 KB
constexpr int kDiagSmemBytes = kDiagStages * kDiagStageBytes + 1024;  // + alignment
constexpr int kDiagTmemCols = kBM;
constexpr uint32_t kIdescDiag = idesc_tf32(kBM, kBM);
constexpr int kDiagAhead = 2;  // a group's steps in registers

struct DiagArgs {
  const float* A;       // rows = channels, K-major with stride ld
  int64_t ld, rows;
  const int32_t* idx;   // tile row r reads stored row idx[r]; null: the stored order
  int64_t K;
  int64_t k_chunk;      // blockIdx.y = chunk c covers k in [c * k_chunk, (c + 1) * k_chunk)
  float* out;           // out[c * chunk_stride + (r / 8) * 64 + (r % 8) * 8 + b]
  int64_t chunk_stride;
  float alpha;
  unsigned* err;
};

__global__ void __launch_bounds__(kDiagThreads, 1) syrk_diag_kernel(DiagArgs a) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  extern __shared__ __align__(1024) char smem_raw[];
  char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t full[kDiagStages], empty[kDiagStages], done;
  __shared__ uint32_t tmem_slot;
  __shared__ float blk[kBM][9];   // each tile row: the 8 entries of its own block row
  __shared__ int32_t src[kBM];    // stored row of each tile row (-1 past the end or out of range)

  const int64_t m0 = (int64_t)blockIdx.x * kBM;
  const int64_t kbeg = (int64_t)blockIdx.y * a.k_chunk;
  const int64_t kend = min(a.K, kbeg + a.k_chunk);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < kBM) {
    const int64_t r = m0 + tid;
    int32_t p = -1;
    if (r < a.rows) {
      p = a.idx ? a.idx[r] : (int32_t)r;
      if (p < 0 || p >= a.rows) {
        raise_error(a.err, ERRBIT_INDEX);
        p = -1;
      }
    }
    src[tid] = p;
  }
  if (warp == 0) tmem_alloc(&tmem_slot, kDiagTmemCols);
  if (tid == 0) {
    for (int s = 0; s < kDiagStages; ++s) {
      mbar_init(smem_u32(&full[s]), kBM);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    mbar_init(smem_u32(&done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  const int nkt = (int)((kend - kbeg + kBK - 1) / kBK);
  bool ok = true;
  if (warp < kDiagStages * 4) {
    // Group w fills stage w with the steps w, w + 4, ...; a thread's values come kDiagAhead of its
    // steps early.
    const int w = warp >> 2, r = tid & (kBM - 1);
    const float* row = src[r] >= 0 ? a.A + src[r] * a.ld : nullptr;
    const bool aligned = (a.ld & 3) == 0 && ((uintptr_t)a.A & 15) == 0;
    auto load = [&](int kt, float v[kBK]) {
      const int64_t k = kbeg + (int64_t)kt * kBK;
      load_row(row ? row + k : nullptr, kend - k, aligned, v);
    };
    char* hi = smem + w * kDiagStageBytes;
    char* lo = hi + kAStageBytes;
    float va[kDiagAhead][kBK];
#pragma unroll
    for (int u = 0; u < kDiagAhead; ++u)
      if (w + u * kDiagStages < nkt) load(w + u * kDiagStages, va[u]);
    for (int j0 = 0; w + j0 * kDiagStages < nkt && ok; j0 += kDiagAhead) {
#pragma unroll
      for (int u = 0; u < kDiagAhead; ++u) {
        const int j = j0 + u, kt = w + j * kDiagStages;
        if (kt >= nkt || !ok) break;
        if (j > 0) ok = mbar_wait(smem_u32(&empty[w]), (uint32_t)((j - 1) & 1), a.err);
        if (!ok) break;
        split_store(va[u], r, hi, lo);
        if (kt + kDiagAhead * kDiagStages < nkt) load(kt + kDiagAhead * kDiagStages, va[u]);
        fence_async_smem();
        mbar_arrive(smem_u32(&full[w]));
      }
    }
  } else if (lane == 0) {
    for (int kt = 0; kt < nkt && ok; ++kt) {
      const int s = kt % kDiagStages;
      ok = mbar_wait(smem_u32(&full[s]), (uint32_t)((kt / kDiagStages) & 1), a.err);
      if (!ok) break;
      tc_fence_after();
      const uint32_t hi = smem_u32(smem + s * kDiagStageBytes), lo = hi + kAStageBytes;
      constexpr uint32_t sbo = (kBK / 4) * 128;
#pragma unroll
      for (int ks = 0; ks < kBK / 8; ++ks) {
        const uint64_t dh = smem_desc(hi + ks * 256, 128, sbo);
        const uint64_t dl = smem_desc(lo + ks * 256, 128, sbo);
        // same order as the dense tile: hi.hi, hi.lo, lo.hi
        mma_tf32(tmem, dh, dh, kIdescDiag, (kt > 0 || ks > 0) ? 1u : 0u);
        mma_tf32(tmem, dh, dl, kIdescDiag, 1u);
        mma_tf32(tmem, dl, dh, kIdescDiag, 1u);
      }
      mma_commit(smem_u32(&empty[s]));
    }
    mma_commit(smem_u32(&done));  // (after a timeout too: the MMAs issued so far)
  }
  __syncwarp();
  ok = mbar_wait(smem_u32(&done), 0u, a.err) && ok;
  ok = __syncthreads_and(ok);
  tc_fence_after();

  const int row = tid;  // the first 128 threads
  if (ok && warp < 4) {
    // the warp's rows meet their block partners in columns [32 warp, 32 warp + 32)
    float v[32];
    tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(warp * 32), v);
    const int q = lane >> 3;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float x = v[j];
#pragma unroll
      for (int qq = 1; qq < 4; ++qq)
        if (q == qq) x = v[8 * qq + j];
      blk[row][j] = x;
    }
  }
  __syncthreads();
  if (ok && warp < 4 && m0 + row < a.rows && src[row] >= 0) {
    const int ra = row & 7, g0 = row & ~7;
    const int32_t pa = src[row];
    float* o = a.out + (int64_t)blockIdx.y * a.chunk_stride + (m0 + row) * 8;
    float w[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const int32_t pb = src[g0 + b];
      w[b] = a.alpha * (pa <= pb ? blk[row][b] : blk[g0 + b][ra]);
    }
    *reinterpret_cast<float4*>(o) = make_float4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<float4*>(o + 4) = make_float4(w[4], w[5], w[6], w[7]);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kDiagTmemCols);
}

}  // namespace tc
}  // namespace crvq
