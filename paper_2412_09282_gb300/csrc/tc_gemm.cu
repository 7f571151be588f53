// The tcgen05 3xTF32 products: the image-fed kernel (dense X^T X, the sums of the losses, the coupled
// sweep's blocks) and the host side of the diagonal blocks alone (tc_gemm.cuh). The tensor core
// accumulates fp32 with a small systematic rounding bias per accumulation step, so K is cut into
// chunks of at most kKChunk and the few chunk partials of an element are summed afterwards in fp32,
// in chunk order (a relative error of a few u); squares are summed per row in fp32 and per tile in
// fp64.
#include <algorithm>

#include "common.cuh"
#include "img.cuh"
#include "kernels.h"
#include "tc_gemm.cuh"

namespace crvq {

namespace {

constexpr int64_t kKChunk = 1024;

// scale * sum_c P[c * stride + e], chunks in order (the one rounding sequence every split-K
// product of this file uses, so its dense and block-only forms agree bit for bit)
__device__ __forceinline__ float chunk_sum(const float* __restrict__ P, int chunks,
                                           int64_t stride, int64_t e, float scale) {
  float s = 0.f;
  for (int c = 0; c < chunks; ++c) s += P[c * stride + e];
  return s * scale;
}

// S = scale * the sum of the chunk partials P[c] (N x N each), and its diagonal.
__global__ void __launch_bounds__(256)
sum_partials_kernel(const float* __restrict__ P, int64_t N, int chunks, float scale,
                    float* __restrict__ S, float* __restrict__ diag) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N * N;
       e += (int64_t)gridDim.x * blockDim.x) {
    const float v = chunk_sum(P, chunks, N * N, e, scale);
    S[e] = v;
    if (e % (N + 1) == 0) diag[e / (N + 1)] = v;
  }
}

// Original-order blocks without the damping, and their diagonal xsq.
__global__ void __launch_bounds__(256)
blocks_sum_kernel(const float* __restrict__ P, int chunks, int64_t stride, float scale, int64_t N,
                  float* __restrict__ xsq, float* __restrict__ Hb) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N * 8;
       e += (int64_t)gridDim.x * blockDim.x) {
    const float v = chunk_sum(P, chunks, stride, e, scale);
    Hb[e] = v;
    if (((e >> 3) & 7) == (e & 7)) xsq[e >> 3] = v;
  }
}

// Adds delta to the diagonals of the original-order blocks (rounded once from fp64, as the dense path
// does).
__global__ void __launch_bounds__(256)
blocks_add_delta_kernel(const float* __restrict__ xsq, int64_t N, const double* __restrict__ delta64,
                        float* __restrict__ Hb) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) Hb[i * 8 + (i & 7)] = (float)((double)xsq[i] + *delta64);
}

// blocks_sum_kernel, hessian_delta_kernel and blocks_add_delta_kernel in one block, the same values, for
// up to kSmallRows channels and kSmallTerms chunk terms: there two launches more are most of the difference
// (16 x 128: 32 us as three kernels, 28 as one; 1024 x 512 44 us either way; with 32768 terms, 4096 x
// 1024, one block is slower, 54 us instead of 51).
constexpr int kSmallRows = 1024;
constexpr int64_t kSmallTerms = 8192;

__global__ void __launch_bounds__(kSmallRows)
blocks_small_kernel(const float* __restrict__ P, int chunks, int64_t stride, float scale, int N,
                    float damp_rel, float* __restrict__ xsq, float* __restrict__ delta_out,
                    double* __restrict__ delta64, float* __restrict__ Hb) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  __shared__ double part[kSmallRows];
  __shared__ float sx[kSmallRows];
  const int t = threadIdx.x;
  for (int e = t; e < N * 8; e += kSmallRows) {
    const float v = chunk_sum(P, chunks, stride, e, scale);
    if (((e >> 3) & 7) == (e & 7))
      xsq[e >> 3] = sx[e >> 3] = v;
    else
      Hb[e] = v;
  }
  __syncthreads();
  part[t] = t < N ? (double)sx[t] : 0.0;
  __syncthreads();
  for (int w = kSmallRows / 2; w > 0; w >>= 1) {
    if (t < w) part[t] += part[t + w];
    __syncthreads();
  }
  const double delta = (double)damp_rel * (part[0] / (double)N);
  if (t == 0) {
    if (delta_out) *delta_out = (float)delta;
    *delta64 = delta;
  }
  if (t < N) Hb[t * 8 + (t & 7)] = (float)((double)sx[t] + delta);
}

// Blocks of a given channel order with a known delta.
__global__ void __launch_bounds__(256)
blocks_damp_kernel(const float* __restrict__ P, int chunks, int64_t stride, float scale,
                   int64_t N, const double* __restrict__ delta64, float* __restrict__ Hb) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const double delta = *delta64;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N * 8;
       e += (int64_t)gridDim.x * blockDim.x) {
    const float v = chunk_sum(P, chunks, stride, e, scale);
    Hb[e] = ((e >> 3) & 7) == (e & 7) ? (float)((double)v + delta) : v;
  }
}

// out[a][k] = X[k][a] (X: n x N row-major) for a < N, k < n; columns k in [n, ldt) are 0.
__global__ void __launch_bounds__(256)
transpose_kernel(const float* __restrict__ X, int64_t n, int64_t N, float* __restrict__ out,
                 int64_t ldt) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  __shared__ float t[32][33];
  const int64_t k0 = (int64_t)blockIdx.x * 32, a0 = (int64_t)blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const int64_t k = k0 + r, a = a0 + tx;
    t[r][tx] = (k < n && a < N) ? X[k * N + a] : 0.f;
  }
  __syncthreads();
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const int64_t a = a0 + r, k = k0 + tx;
    if (a < N && k < ldt) out[a * ldt + k] = t[tx][r];
  }
}

}  // namespace

// ---- image-fed 3xTF32 products A B^T
// Both operands are first written once as tf32 hi / lo images in the tcgen05 canonical
// K-major layout (no swizzle): 256-row blocks, 16-column slabs of 16 KB each, slabs of a block
// consecutive. A CTA then computes one 128 x 256 tile with no work of its threads on the
// operand path: warp 0 streams the slabs by bulk copy (TMA) into a four-stage ring, warp 1
// issues the MMAs (hi.hi, hi.lo, lo.hi per 8-column step), and warps 2-5 keep the K-chunk
// partials: after every 1024-column chunk the accumulator is added, in chunk order and in fp32, to
// a running sum kept in the other half of tensor memory. The last chunk's sum goes to the epilogue:
//   kSumsq      the sum of its squares (the full loss of Alg. 1 QuantLoss);
//   kDot        the sum of its products with E's entries in fp32 pairs, in fp64 beyond fp32's range
//               (tr(D H D^T));
//   kSymmetric  C[m][n] = C[n][m] = alpha D[m][n] for n >= m (the Hessian; tiles below the
//               diagonal do nothing);
//   kPlain      C[m][n] = alpha D[m][n] (blockIdx.y: one K chunk each, to its own C).
// Row-major stores go through shared memory, so that a warp writes 128 consecutive bytes of a row.
namespace img {
namespace {

constexpr int kAStage = 2 * (kSlabBytes / 2);      // A hi + lo, 128 rows: 16 KB
constexpr int kBStage = 2 * kSlabBytes;            // B hi + lo, 256 rows: 32 KB
constexpr int kStageBytes = kAStage + kBStage;     // 48 KB
constexpr int kStages = 4;
constexpr int kStageOut = 4 * 32 * 33 * 4;         // transposing buffers of the storing warps
constexpr int kSmem = kStages * kStageBytes + kStageOut + 1024 + 256;
constexpr int kThreads = 192;
constexpr int kChunkSlabs = 1024 / kSlabK;         // slabs per K chunk
constexpr uint32_t kIdesc = tc::idesc_tf32(128, 256);

// hi / lo images of four values at (r, k).
__device__ __forceinline__ void put_image(const float v[4], int64_t r, int64_t k, int64_t nslab, char* hi,
                                          char* lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    h[j] = tc::to_tf32(v[j]);
    l[j] = tc::to_tf32(v[j] - __uint_as_float(h[j]));
  }
  const int64_t off = img_off(r, k, nslab);
  *reinterpret_cast<uint4*>(hi + off) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4*>(lo + off) = make_uint4(l[0], l[1], l[2], l[3]);
}

// Images of src[r][cols[k]] with whole rows staged in shared memory, kGatherRows at a time: every
// row is read once and in order. (image_kernel's four-byte reads fetch a 32-byte sector each: the two
// images of a 4096 x 4096 loss over 4096 tokens took 125 us, now 92.)
// Entries outside [0, K) read as 0, the padding is zeros, as in image_kernel.
constexpr int kGatherRows = 4;
constexpr size_t kGatherSmem = 200 * 1024;  // the largest staging

__global__ void __launch_bounds__(512)
image_gather_kernel(const float* __restrict__ src, const int32_t* __restrict__ cols, int64_t rows,
                    int64_t K, int64_t rows_pad, int64_t nslab, char* __restrict__ hi,
                    char* __restrict__ lo) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  extern __shared__ __align__(16) float staged[];  // [kGatherRows][K]
  const bool vec = (K & 3) == 0 && ((uintptr_t)src & 15) == 0;
  const int r = threadIdx.x % kGatherRows;
  for (int64_t r0 = (int64_t)blockIdx.x * kGatherRows; r0 < rows_pad;
       r0 += (int64_t)gridDim.x * kGatherRows) {
    const int64_t n = max((int64_t)0, min((int64_t)kGatherRows, rows - r0)) * K;
    __syncthreads();  // the rows before have been written
    if (vec) {
      for (int64_t e = (int64_t)threadIdx.x * 4; e < n; e += blockDim.x * 4)
        *reinterpret_cast<float4*>(staged + e) =
            __ldg(reinterpret_cast<const float4*>(src + r0 * K + e));
    } else {
      for (int64_t e = threadIdx.x; e < n; e += blockDim.x) staged[e] = src[r0 * K + e];
    }
    __syncthreads();
    for (int64_t q = threadIdx.x / kGatherRows; q < nslab * (kSlabK / 4);
         q += blockDim.x / kGatherRows) {
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t k = 4 * q + j;
        const int32_t c = k < K ? cols[k] : -1;
        v[j] = r0 + r < rows && c >= 0 && c < K ? staged[r * K + c] : 0.f;
      }
      put_image(v, r0 + r, 4 * q, nslab, hi, lo);
    }
  }
}

// One warp = 8 rows x one 16-column slab: reads 8 x 64 B, writes 512 contiguous bytes per
// image. Element (r, k) is src[r][k] - sub[r][k] (sub optional, same layout), or
// src[r][cols[k]] with a column order (entries outside [0, K) read as 0; the caller checks
// the order). Rows >= rows and columns >= K are written as zeros (the images' padding).
__global__ void __launch_bounds__(256)
image_kernel(const float* __restrict__ src, const float* __restrict__ sub,
             const int32_t* __restrict__ cols, int64_t rows, int64_t K, int64_t ld,
             int64_t rows_pad, int64_t nslab, char* __restrict__ hi, char* __restrict__ lo) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r = (int64_t)blockIdx.x * 8 + (lane & 7);
  const int64_t sl = (int64_t)blockIdx.y * 8 + warp;
  if (sl >= nslab || r >= rows_pad) return;
  const int64_t k = sl * kSlabK + (lane >> 3) * 4;
  float v[4] = {0.f, 0.f, 0.f, 0.f};
  if (r < rows) {
    const float* p = src + r * ld;
    if (cols) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int32_t c = (k + j < K) ? cols[k + j] : -1;
        v[j] = (c >= 0 && c < K) ? p[c] : 0.f;
      }
    } else if (k + 4 <= K && (ld & 3) == 0 && ((uintptr_t)src & 15) == 0 &&
               (!sub || ((uintptr_t)sub & 15) == 0)) {
      const float4 x = __ldg(reinterpret_cast<const float4*>(p + k));
      v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
      if (sub) {
        const float4 y = __ldg(reinterpret_cast<const float4*>(sub + r * ld + k));
        v[0] -= y.x; v[1] -= y.y; v[2] -= y.z; v[3] -= y.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        v[j] = (k + j < K) ? (sub ? p[k + j] - sub[r * ld + k + j] : p[k + j]) : 0.f;
    }
  }
  put_image(v, r, k, nslab, hi, lo);
}

// Images of X^T: element (r, k) is X[k][r] (X: K x rows row-major). A thread takes row r, four
// columns: its reads are 128 consecutive bytes per warp, its writes whole 128-byte core matrices.
__global__ void __launch_bounds__(256)
image_t_kernel(const float* __restrict__ X, int64_t rows, int64_t K, int64_t rows_pad,
               int64_t nslab, char* __restrict__ hi, char* __restrict__ lo) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const int64_t r = (int64_t)blockIdx.x * 32 + (threadIdx.x & 31);
  if (r >= rows_pad) return;
  for (int64_t k = ((int64_t)blockIdx.y * 8 + (threadIdx.x >> 5)) * 4; k < nslab * kSlabK;
       k += (int64_t)gridDim.y * 32) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float v = (r < rows && k + j < K) ? __ldg(X + (k + j) * rows + r) : 0.f;
      h[j] = tc::to_tf32(v);
      l[j] = tc::to_tf32(v - __uint_as_float(h[j]));
    }
    const int64_t off = img_off(r, k, nslab);
    *reinterpret_cast<uint4*>(hi + off) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(lo + off) = make_uint4(l[0], l[1], l[2], l[3]);
  }
}

enum Epilogue { kSumsq, kDot, kSymmetric, kPlain };

struct ImgArgs {
  const char *a_hi, *a_lo, *b_hi, *b_lo;  // images
  int64_t nslab;                          // slabs per block (both images)
  int64_t slabs_y;                        // slabs per blockIdx.y (nslab, or one K chunk)
  int tiles_n;                            // 256-row tiles of B
  double* part;                           // kSumsq, kDot: part[tile]
  const float* E;                         // kDot: E[m][n]
  float* C;                               // kSymmetric, kPlain: + blockIdx.y * c_stride
  int64_t ldc, c_stride;                  // leading dimension of C (or E)
  float alpha;
  float* diag;                            // kSymmetric: the diagonal, or null
  int64_t rows_m, rows_n;
  unsigned* err;
};

__device__ __forceinline__ void pair_acc(float& h, float& l, float x) {  // (h, l) += x
  const float s = __fadd_rn(h, x);
  const float bp = __fsub_rn(s, h);
  l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, bp)), __fsub_rn(x, bp)));
  h = s;
}

template <int EPI>
__global__ void __launch_bounds__(kThreads, 1) img_gemm_kernel(ImgArgs a) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  extern __shared__ __align__(1024) char smem_raw[];
  char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  float* stage_out = reinterpret_cast<float*>(smem + kStages * kStageBytes);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes + kStageOut);
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
  __shared__ double red[4];
  __shared__ int ok_s[3];

  const int tile = blockIdx.x;
  const int bm = tile / a.tiles_n, bn = tile % a.tiles_n;
  if (EPI == kSymmetric && (int64_t)(bn + 1) * 256 <= (int64_t)bm * 128) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t slab0 = (int64_t)blockIdx.y * a.slabs_y;
  const int64_t nslab = min(a.slabs_y, a.nslab - slab0);  // of this CTA
  const int nchunk = (int)((nslab + kChunkSlabs - 1) / kChunkSlabs);

  if (warp == 0) tc::tmem_alloc(tmem_slot, 512);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(tc::smem_u32(&full[s]), 1);
      tc::mbar_init(tc::smem_u32(&empty[s]), 1);
    }
    tc::mbar_init(tc::smem_u32(acc_full), 1);
    tc::mbar_init(tc::smem_u32(acc_empty), 128);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 3) ok_s[threadIdx.x] = 1;
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;   // columns [0, 256): accumulator; [256, 512): chunk sum

  if (warp == 0) {
    if (lane == 0) {  // producer
      const int64_t a0 = ((int64_t)(bm >> 1) * a.nslab + slab0) * kSlabBytes + (bm & 1) * (kSlabBytes / 2);
      const int64_t b0 = ((int64_t)bn * a.nslab + slab0) * kSlabBytes;
      const char *ah = a.a_hi + a0, *al = a.a_lo + a0, *bh = a.b_hi + b0, *bl = a.b_lo + b0;
      bool ok = true;
      int64_t it = 0;
      for (; it < nslab; ++it) {
        const int s = (int)(it % kStages);
        if (it >= kStages)
          ok = tc::mbar_wait(tc::smem_u32(&empty[s]), (uint32_t)((it / kStages - 1) & 1), a.err);
        if (!ok) break;
        char* st = smem + s * kStageBytes;
        const uint32_t fb = tc::smem_u32(&full[s]);
        tc::mbar_expect_tx(fb, kStageBytes);
        tc::bulk_copy_g2s(tc::smem_u32(st), ah + it * kSlabBytes, kSlabBytes / 2, fb);
        tc::bulk_copy_g2s(tc::smem_u32(st + kSlabBytes / 2), al + it * kSlabBytes, kSlabBytes / 2, fb);
        tc::bulk_copy_g2s(tc::smem_u32(st + kAStage), bh + it * kSlabBytes, kSlabBytes, fb);
        tc::bulk_copy_g2s(tc::smem_u32(st + kAStage + kSlabBytes), bl + it * kSlabBytes, kSlabBytes, fb);
      }
      // No copy may land in this block's shared memory after its end: the last ones are waited for here
      // (bounded), whether or not a timeout kept the MMAs from waiting for them.
      for (int64_t u = it > kStages ? it - kStages : 0; u < it; ++u)
        ok = tc::mbar_wait(tc::smem_u32(&full[u % kStages]), (uint32_t)((u / kStages) & 1), a.err) && ok;
      if (!ok) ok_s[0] = 0;
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer
      bool ok = true;
      for (int64_t it = 0; it < nslab && ok; ++it) {
        const int s = (int)(it % kStages);
        const int64_t c = it / kChunkSlabs;
        const bool first = (it % kChunkSlabs) == 0;
        if (first && c > 0) ok = tc::mbar_wait(tc::smem_u32(acc_empty), (uint32_t)((c - 1) & 1), a.err);
        if (ok) ok = tc::mbar_wait(tc::smem_u32(&full[s]), (uint32_t)((it / kStages) & 1), a.err);
        if (!ok) break;
        tc::tc_fence_after();
        const uint32_t st = tc::smem_u32(smem + s * kStageBytes);
        constexpr uint32_t sbo = (kSlabK / 4) * 128;
#pragma unroll
        for (int ks = 0; ks < kSlabK / 8; ++ks) {
          const uint32_t koff = ks * 256;
          const uint64_t dah = tc::smem_desc(st + koff, 128, sbo);
          const uint64_t dal = tc::smem_desc(st + kSlabBytes / 2 + koff, 128, sbo);
          const uint64_t dbh = tc::smem_desc(st + kAStage + koff, 128, sbo);
          const uint64_t dbl = tc::smem_desc(st + kAStage + kSlabBytes + koff, 128, sbo);
          tc::mma_tf32(tmem, dah, dbh, kIdesc, (first && ks == 0) ? 0u : 1u);
          tc::mma_tf32(tmem, dah, dbl, kIdesc, 1u);
          tc::mma_tf32(tmem, dal, dbh, kIdesc, 1u);
        }
        tc::mma_commit(tc::smem_u32(&empty[s]));
        if ((it % kChunkSlabs) == kChunkSlabs - 1 || it == nslab - 1)
          tc::mma_commit(tc::smem_u32(acc_full));
      }
      if (!ok) ok_s[1] = 0;
    }
  } else {  // warps 2-5: one accumulator row (tensor-memory lane) per thread
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const int64_t m0 = (int64_t)bm * 128 + (warp & 3) * 32, m = m0 + lane;
    float* C = EPI == kPlain || EPI == kSymmetric ? a.C + blockIdx.y * a.c_stride : nullptr;
    float* so = stage_out + (warp & 3) * 32 * 33;
    float sq = 0.f, sl = 0.f;  // kSumsq: the sum of squares; kDot: a pair
    double beyond = 0.0;       // kDot: runs of 32 products that leave fp32's range
    bool ok = true;
    for (int c = 0; c < nchunk && ok; ++c) {
      ok = tc::mbar_wait(tc::smem_u32(acc_full), (uint32_t)(c & 1), a.err);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc::tc_fence_after();
      const bool last = c == nchunk - 1;
#pragma unroll 1
      for (int c0 = 0; c0 < 256; c0 += 32) {
        uint32_t v[32], w[32];
        float e[EPI == kDot ? 32 : 1];  // E's entries of this lane's column, all in flight at once
        if (EPI == kDot && last) {
          const int64_t n = min((int64_t)bn * 256 + c0 + lane, a.rows_n - 1);
#pragma unroll
          for (int r = 0; r < 32; ++r) e[r & (EPI == kDot ? 31 : 0)] = __ldg(a.E + min(m0 + r, a.rows_m - 1) * a.ldc + n);
        }
        tc::tmem_ld32_nowait(tmem + lane_base + (uint32_t)c0, v);
        tc::tmem_wait_ld_dep(v);
        if (c > 0) {
          tc::tmem_ld32_nowait(tmem + lane_base + 256u + (uint32_t)c0, w);
          tc::tmem_wait_ld_dep(w);
#pragma unroll
          for (int j = 0; j < 32; ++j)
            v[j] = __float_as_uint(__fadd_rn(__uint_as_float(w[j]), __uint_as_float(v[j])));
        }
        if (last && EPI == kSumsq) {
#pragma unroll
          for (int j = 0; j < 32; ++j) sq = fmaf(__uint_as_float(v[j]), __uint_as_float(v[j]), sq);
        } else if (last) {
          // rows of 32 columns: registers hold a row per lane, memory wants a row per warp
          const int64_t n0 = (int64_t)bn * 256 + c0, n = n0 + lane;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float x = EPI == kDot ? __uint_as_float(v[j]) : a.alpha * __uint_as_float(v[j]);
            so[lane * 33 + j] = x;
            if (EPI == kSymmetric && n0 + j > m && m < a.rows_m && n0 + j < a.rows_n)
              C[(n0 + j) * a.ldc + m] = x;
            if (EPI == kSymmetric && a.diag && n0 + j == m && m < a.rows_m) a.diag[m] = x;
          }
          __syncwarp();
          if (EPI == kDot) {
            const float sq0 = sq, sl0 = sl;
#pragma unroll
            for (int r = 0; r < 32; ++r) {  // (operand padding makes x zero past the rows of A and B)
              const float x = so[r * 33 + lane], er = e[r & (EPI == kDot ? 31 : 0)];
              const float p = __fmul_rn(x, er);
              pair_acc(sq, sl, p);
              sl = __fadd_rn(sl, __fmaf_rn(x, er, -p));
            }
            if (!isfinite(sq) || !isfinite(sl)) {
              sq = sq0;
              sl = sl0;
#pragma unroll
              for (int r = 0; r < 32; ++r)
                beyond += (double)so[r * 33 + lane] * (double)e[r & (EPI == kDot ? 31 : 0)];
            }
          } else if (n < a.rows_n) {
#pragma unroll 8
            for (int r = 0; r < 32; ++r) {
              const int64_t mr = m0 + r;
              if (mr >= a.rows_m) break;
              if (EPI == kPlain || n >= mr) C[mr * a.ldc + n] = so[r * 33 + lane];
            }
          }
          __syncwarp();
        } else {
          tc::tmem_st32_wait(tmem + lane_base + 256u + (uint32_t)c0, v);
        }
      }
      tc::tc_fence_before();
      if (!last) tc::mbar_arrive(tc::smem_u32(acc_empty));
    }
    if (!ok) sq = sl = 0.f;
    double sd = (double)sq + (double)sl + (EPI == kDot && ok ? beyond : 0.0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sd += __shfl_xor_sync(0xffffffffu, sd, o);
    if (lane == 0) red[warp - 2] = sd;
    if (lane == 0 && !ok) ok_s[2] = 0;
  }
  tc::tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && (EPI == kSumsq || EPI == kDot)) {
    const bool ok = ok_s[0] && ok_s[1] && ok_s[2];
    a.part[tile] = ok ? ((red[0] + red[1]) + (red[2] + red[3])) : 0.0;
  }
  if (warp == 0) {
    __syncwarp();
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 512);
  }
}

template <int EPI>
crvq_status launch(const ImgArgs& a, int64_t tiles_m, int64_t chunks, cudaStream_t stream) {
  CRVQ_TRY(smem_limit((const void*)img_gemm_kernel<EPI>, kSmem));
  CRVQ_CUDA(launch_pdl(img_gemm_kernel<EPI>, dim3((unsigned)(tiles_m * a.tiles_n),
                       (unsigned)chunks), dim3(kThreads), kSmem, stream, a));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

int64_t pad_rows(int64_t rows) { return ceil_div(rows, (int64_t)kRowsBlk) * kRowsBlk; }

}  // namespace
}  // namespace img

size_t img_bytes(int64_t rows, int64_t K) {
  return (size_t)img::pad_rows(rows) * ceil_div(K, (int64_t)img::kSlabK) * img::kSlabK * 4;
}

int64_t img_k_chunks(int64_t K) { return std::max<int64_t>(1, ceil_div(K, kKChunk)); }

crvq_status launch_images(const float* src, const float* sub, const int32_t* cols, int64_t rows,
                          int64_t K, char* hi, char* lo, cudaStream_t stream) {
  const int64_t nslab = ceil_div(K, (int64_t)img::kSlabK), pad = img::pad_rows(rows);
  const size_t staged = (size_t)img::kGatherRows * K * sizeof(float);
  if (cols && staged <= img::kGatherSmem) {
    CRVQ_TRY(smem_limit((const void*)img::image_gather_kernel, img::kGatherSmem));
    const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(4, (int64_t)(220 * 1024 / (staged + 1024))));
    CRVQ_CUDA(launch_pdl(img::image_gather_kernel, dim3((unsigned)std::min<int64_t>(pad /
                         img::kGatherRows, per_sm * sm_count())), dim3(512), staged, stream, src,
                         cols, rows, K, pad, nslab, hi, lo));
    CRVQ_LAUNCHED();
    return CRVQ_OK;
  }
  CRVQ_CUDA(launch_pdl(img::image_kernel, dim3((unsigned)(pad / 8), (unsigned)ceil_div(nslab, 8)),
                       dim3(256), 0, stream, src, sub, cols, rows, K, K, pad, nslab, hi, lo));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

// S = X^T X / n (X: n x N row-major) into S (N x N), both triangles, and its diagonal: the images of X^T, then one
// product over the tiles that reach the upper triangle, chunk sums kept in tensor memory. (Splitting
// the operands in the product's own shared-memory stages bound it by the L1TEX pipe: 765 us at
// N = n = 4096, with 57 us more for adding chunk partials kept in memory; now 317 us in all.)
crvq_status launch_tc_syrk(const float* X, int64_t n, int64_t N, float* S, float* diag,
                           cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  const size_t bytes = img_bytes(N, n);
  Scratch mem;
  CRVQ_TRY(mem.alloc(2 * bytes, stream));
  char *hi = mem.as<char>(), *lo = hi + bytes;
  const int64_t nslab = ceil_div(n, (int64_t)img::kSlabK), pad = img::pad_rows(N);
  {
    ProfScope ps("hessian_images", stream, 12.0 * (double)n * N);
    const unsigned gy = (unsigned)std::min<int64_t>(ceil_div(nslab * 4, 8), 65535);
    CRVQ_CUDA(launch_pdl(img::image_t_kernel, dim3((unsigned)(pad / 32), gy), dim3(256), 0, stream,
                         X, N, n, pad, nslab, hi, lo));
    CRVQ_LAUNCHED();
  }
  // Few tiles (small N): each K chunk in its own CTA, the partials added afterwards in chunk order;
  // otherwise a CTA runs through all chunks of its tile. The same rounding sequence.
  const int64_t tiles_m = ceil_div(N, (int64_t)128), tiles_n = ceil_div(N, (int64_t)256);
  const int64_t chunks = img_k_chunks(n);
  const bool split = chunks > 1 && tiles_m * tiles_n <= sm_count();
  const float scale = (float)(1.0 / (double)n);
  Scratch pmem;
  if (split) CRVQ_TRY(pmem.alloc((size_t)chunks * N * N * sizeof(float), stream));
  img::ImgArgs g{};
  g.a_hi = g.b_hi = hi;
  g.a_lo = g.b_lo = lo;
  g.nslab = nslab;
  g.slabs_y = split ? img::kChunkSlabs : nslab;
  g.tiles_n = (int)tiles_n;
  g.C = split ? pmem.as<float>() : S;
  g.ldc = N;
  g.c_stride = N * N;
  g.alpha = split ? 1.f : scale;
  g.diag = split ? nullptr : diag;
  g.rows_m = g.rows_n = N;
  g.err = err;
  {
    ProfScope ps("hessian_gemm_tc", stream, 2.0 * (double)n * N * N);
    CRVQ_TRY(img::launch<img::kSymmetric>(g, tiles_m, split ? chunks : 1, stream));
  }
  if (split) {
    ProfScope ps("hessian_sum_partials", stream, (double)chunks * N * N * 4.0);
    const int blocks = (int)std::min<int64_t>(ceil_div(N * N, 256), 16 * sm_count());
    CRVQ_CUDA(launch_pdl(sum_partials_kernel, dim3(blocks), dim3(256), 0, stream, pmem.as<float>(),
                         N, (int)chunks, scale, S, diag));
    CRVQ_LAUNCHED();
  }
  return CRVQ_OK;
}

// part[0 .. nparts) = partial sums of ||(A - A_sub) B'^T||_F^2 with A, A_sub: M x K, B: Nb x K
// (row-major, leading dimension K; B' = B with columns in the order B_cols when given), one
// per 128 x 256 tile; part_cap must hold ceil(M / 128) * ceil(Nb / 256) values. Returns the
// number of partials written.
crvq_status launch_tc_sumsq(const float* A, const float* A_sub, int64_t M, const float* B,
                            const int32_t* B_cols, int64_t Nb, int64_t K, double* part,
                            int64_t part_cap, int64_t* nparts, cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  const int64_t tiles_m = ceil_div(M, (int64_t)128), tiles_n = ceil_div(Nb, (int64_t)256);
  if (tiles_m * tiles_n > part_cap)
    return fail(CRVQ_ERR_UNSUPPORTED, "loss product: %lld tiles exceed %lld partials",
                (long long)(tiles_m * tiles_n), (long long)part_cap);
  if (tiles_m * tiles_n > INT32_MAX)
    return fail(CRVQ_ERR_UNSUPPORTED, "loss product: too many tiles");
  const size_t a_bytes = img_bytes(M, K), b_bytes = img_bytes(Nb, K);
  Scratch mem;
  CRVQ_TRY(mem.alloc(2 * a_bytes + 2 * b_bytes, stream));
  char* a_hi = mem.as<char>();
  char* a_lo = a_hi + a_bytes;
  char* b_hi = a_lo + a_bytes;
  char* b_lo = b_hi + b_bytes;
  {
    ProfScope ps("loss_images", stream, 12.0 * (double)(M + Nb) * K);
    CRVQ_TRY(launch_images(A, A_sub, nullptr, M, K, a_hi, a_lo, stream));
    CRVQ_TRY(launch_images(B, nullptr, B_cols, Nb, K, b_hi, b_lo, stream));
  }
  img::ImgArgs g{};
  g.a_hi = a_hi;
  g.a_lo = a_lo;
  g.b_hi = b_hi;
  g.b_lo = b_lo;
  g.nslab = g.slabs_y = ceil_div(K, (int64_t)img::kSlabK);
  g.tiles_n = (int)tiles_n;
  g.part = part;
  g.err = err;
  ProfScope ps("loss_gemm_tc", stream, 2.0 * (double)M * Nb * K);
  CRVQ_TRY(img::launch<img::kSumsq>(g, tiles_m, 1, stream));
  *nparts = tiles_m * tiles_n;
  return CRVQ_OK;
}

// P[c][m][n] = the K chunk c of A B^T (A: M rows starting at block row `a_row0`, a multiple of 256,
// of its image; B: Nb rows; both with K columns), c < img_k_chunks(K), each M x Nb.
crvq_status launch_img_gemm_chunks(const char* a_hi, const char* a_lo, int64_t a_row0, int64_t M,
                                   const char* b_hi, const char* b_lo, int64_t Nb, int64_t K,
                                   float* P, cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  const int64_t nslab = ceil_div(K, (int64_t)img::kSlabK);
  const int64_t a_off = a_row0 / img::kRowsBlk * nslab * img::kSlabBytes;
  img::ImgArgs g{};
  g.a_hi = a_hi + a_off;
  g.a_lo = a_lo + a_off;
  g.b_hi = b_hi;
  g.b_lo = b_lo;
  g.nslab = nslab;
  g.slabs_y = img::kChunkSlabs;
  g.tiles_n = (int)ceil_div(Nb, (int64_t)256);
  g.C = P;
  g.ldc = Nb;
  g.c_stride = M * Nb;
  g.alpha = 1.f;
  g.rows_m = M;
  g.rows_n = Nb;
  g.err = err;
  ProfScope ps("gemm_nt_tc", stream, 2.0 * (double)M * Nb * K);
  return img::launch<img::kPlain>(g, ceil_div(M, (int64_t)128), img_k_chunks(K), stream);
}

// part[tile] = partial sums of sum_{m,n} (A B^T)[m][n] E[m][n] (A: M x K, B: Nb x K images; E
// row-major M x Nb), one per 128 x 256 tile.
crvq_status launch_img_dot(const char* a_hi, const char* a_lo, int64_t M, const char* b_hi,
                           const char* b_lo, int64_t Nb, int64_t K, const float* E, double* part,
                           cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  img::ImgArgs g{};
  g.a_hi = a_hi;
  g.a_lo = a_lo;
  g.b_hi = b_hi;
  g.b_lo = b_lo;
  g.nslab = g.slabs_y = ceil_div(K, (int64_t)img::kSlabK);
  g.tiles_n = (int)ceil_div(Nb, (int64_t)256);
  g.part = part;
  g.E = E;
  g.ldc = Nb;
  g.rows_m = M;
  g.rows_n = Nb;
  g.err = err;
  ProfScope ps("coupled_loss", stream, 2.0 * (double)M * Nb * K);
  return img::launch<img::kDot>(g, ceil_div(M, (int64_t)128), 1, stream);
}

crvq_status launch_transpose(const float* X, int64_t n, int64_t N, float* Xt, int64_t ldt,
                             cudaStream_t stream) {
  ProfScope ps("hessian_transpose", stream, 8.0 * (double)n * N);
  CRVQ_CUDA(launch_pdl(transpose_kernel, dim3((unsigned)ceil_div(ldt, 32), (unsigned)ceil_div(N,
                       32)), dim3(256), 0, stream, X, n, N, Xt, ldt));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

// Diagonal 8 x 8 blocks of X^T X / n (+ delta I) for the channel order `perm` (NULL = the
// stored order), from Xt = X^T (N x ldt, ldt a multiple of 4). delta_known: delta64 (fp64) is
// read; otherwise perm must be NULL and xsq, delta (float, may be NULL) and delta64 are
// written. The entries equal those of launch_tc_syrk's dense S plus the damping bit for bit.
crvq_status launch_tc_hessian_blocks(const float* Xt, int64_t ldt, int64_t n, int64_t N,
                                     const int32_t* perm, bool delta_known, float damp_rel,
                                     float* xsq, float* delta, double* delta64, float* Hb,
                                     cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  static bool attr_set[64] = {};
  int dev = 0;
  CRVQ_CUDA(cudaGetDevice(&dev));
  if (dev < 64 && !attr_set[dev]) {
    CRVQ_CUDA(cudaFuncSetAttribute(tc::syrk_diag_kernel,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   tc::kDiagSmemBytes));
    attr_set[dev] = true;
  }
  const int64_t chunks = std::max<int64_t>(1, ceil_div(n, kKChunk));
  const int64_t stride = N * 8;
  Scratch mem;
  CRVQ_TRY(mem.alloc((size_t)chunks * stride * sizeof(float), stream));
  tc::DiagArgs a{};
  a.A = Xt;
  a.ld = ldt;
  a.rows = N;
  a.idx = perm;
  a.K = n;
  a.k_chunk = kKChunk;
  a.out = mem.as<float>();
  a.chunk_stride = stride;
  a.alpha = chunks > 1 ? 1.f : (float)(1.0 / (double)n);
  a.err = err;
  const float scale = chunks > 1 ? (float)(1.0 / (double)n) : 1.f;
  {
    ProfScope ps(perm ? "reorder_blocks_tc" : "hessian_blocks_tc", stream,
                 6.0 * (double)n * N * tc::kBM);
    dim3 grid((unsigned)ceil_div(N, tc::kBM), (unsigned)chunks);
    CRVQ_CUDA(launch_pdl(tc::syrk_diag_kernel, grid, dim3(tc::kDiagThreads), tc::kDiagSmemBytes,
                         stream, a));
    CRVQ_LAUNCHED();
  }
  ProfScope ps("hessian_blocks_finalize", stream, (double)chunks * stride * 4.0);
  if (!delta_known) {
    if (perm) return fail(CRVQ_ERR_UNSUPPORTED, "hessian blocks: delta needs the stored order");
    if (N <= kSmallRows && chunks * stride <= kSmallTerms) {
      CRVQ_CUDA(launch_pdl(blocks_small_kernel, dim3(1), dim3(kSmallRows), 0, stream, mem.as<float>(),
                           (int)chunks, stride, scale, (int)N, damp_rel, xsq, delta, delta64, Hb));
      CRVQ_LAUNCHED();
      return CRVQ_OK;
    }
    const int blocks = (int)std::min<int64_t>(ceil_div(stride, 256), 4 * sm_count());
    CRVQ_CUDA(launch_pdl(blocks_sum_kernel, dim3(blocks), dim3(256), 0, stream, mem.as<float>(),
                         (int)chunks, stride, scale, N, xsq, Hb));
    CRVQ_LAUNCHED();
    CRVQ_TRY(launch_hessian_delta(xsq, N, damp_rel, delta, delta64, stream));
    CRVQ_CUDA(launch_pdl(blocks_add_delta_kernel, dim3((unsigned)ceil_div(N, 256)), dim3(256), 0,
                         stream, xsq, N, delta64, Hb));
  } else {
    const int blocks = (int)std::min<int64_t>(ceil_div(stride, 256), 4 * sm_count());
    CRVQ_CUDA(launch_pdl(blocks_damp_kernel, dim3(blocks), dim3(256), 0, stream, mem.as<float>(),
                         (int)chunks, stride, scale, N, delta64, Hb));
  }
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

}  // namespace crvq
