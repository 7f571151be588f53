// Operand images of the 3xTF32 products (tc_gemm.cu): tf32 hi and lo parts of a row-major matrix in
// the tcgen05 canonical K-major layout (no swizzle), 256-row blocks of 16-column slabs of 16 KB, the
// slabs of a block consecutive.
#pragma once

#include "common.cuh"

namespace crvq {
namespace img {

constexpr int kRowsBlk = 256;                      // image block rows
constexpr int kSlabK = 16;                         // image slab columns
constexpr int kSlabBytes = kRowsBlk * kSlabK * 4;  // 16 KB

// Image byte offset of element (r, k): block r / 256, slab k / 16, then the canonical offset.
__host__ __device__ inline int64_t img_off(int64_t r, int64_t k, int64_t nslab) {
  const int64_t blk = r / kRowsBlk, rr = r % kRowsBlk, sl = k / kSlabK, kk = k % kSlabK;
  return (blk * nslab + sl) * kSlabBytes +
         (((rr >> 3) * (kSlabK / 4) + (kk >> 2)) * 128 + (rr & 7) * 16 + (kk & 3) * 4);
}

}  // namespace img
}  // namespace crvq
