// S1: Hessian proxy H = X^T X / n + delta I (App. A.2; the paper's X is N x O and its proxy
// XX^T is the same matrix as our X^T X).
//
// The dense product X^T X (the crvq_hessian entry) runs on the tensor cores (tc_gemm.cu: tcgen05,
// 3xTF32, tiles that reach the upper triangle, mirrored; 1024-token chunks summed in fp32 in chunk
// order) and writes its diagonal beside it. One CTA sums the diagonal; the damping is added where
// the diagonal blocks are taken. The layer schedule forms only the diagonal blocks
// (launch_tc_hessian_blocks in tc_gemm.cu), with the same values.
#include "common.cuh"
#include "kernels.h"

namespace crvq {

namespace {

// One CTA: delta = damp_rel * mean(xsq) (fixed-order fp64 sum).
__global__ void __launch_bounds__(1024)
hessian_delta_kernel(const float* __restrict__ xsq, int64_t N, float damp_rel,
                     float* __restrict__ delta_out, double* __restrict__ delta64) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  __shared__ double part[1024];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < N; i += blockDim.x) s += (double)xsq[i];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  const double delta = (double)damp_rel * (part[0] / (double)N);
  if (threadIdx.x == 0) {
    if (delta_out) *delta_out = (float)delta;
    *delta64 = delta;
  }
}

// Adds delta to the diagonal of H (rounded once from fp64) and takes the original-order diagonal
// blocks (Hb may be null).
__global__ void __launch_bounds__(256)
hessian_damp_kernel(float* __restrict__ H, int64_t N, const double* __restrict__ delta64,
                    float* __restrict__ Hb) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const double delta = *delta64;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N * kD;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / kD, col = row / kD * kD + e % kD;
    float v = H[row * N + col];
    if (row == col) {
      v = (float)((double)v + delta);
      H[row * N + col] = v;
    }
    if (Hb) Hb[e] = v;
  }
}

__global__ void extract_blocks_kernel(const float* __restrict__ H, int64_t N, int d,
                                      const int32_t* __restrict__ perm,
                                      float* __restrict__ Hb, unsigned* err) {
  pdl_trigger();  // dependents may launch; this grid waits for its predecessor first
  pdl_wait();
  const int64_t G = N / d;
  const int64_t total = G * d * d;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t g = e / (d * d);
    const int r = (int)((e / d) % d), c = (int)(e % d);
    int64_t ra = g * d + r, cb = g * d + c;
    if (perm) {
      ra = perm[ra];
      cb = perm[cb];
      if (ra < 0 || ra >= N || cb < 0 || cb >= N) {
        raise_error(err, ERRBIT_INDEX);
        continue;
      }
    }
    Hb[e] = H[ra * N + cb];
  }
}

}  // namespace

crvq_status launch_hessian_delta(const float* xsq, int64_t N, float damp_rel, float* delta,
                                 double* delta64, cudaStream_t stream) {
  CRVQ_CUDA(launch_pdl(hessian_delta_kernel, dim3(1), dim3(1024), 0, stream, xsq, N, damp_rel,
                       delta, delta64));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

crvq_status launch_hessian(const float* X, int64_t n, int64_t N, int d, float damp_rel,
                           float* H, float* xsq, float* H_blocks, float* delta,
                           cudaStream_t stream) {
  Scratch mem;
  CRVQ_TRY(mem.alloc(sizeof(double), stream));
  CRVQ_TRY(launch_tc_syrk(X, n, N, H, xsq, stream));
  {
    ProfScope ps("hessian_finalize", stream, 0.0);
    CRVQ_TRY(launch_hessian_delta(xsq, N, damp_rel, delta, mem.as<double>(), stream));
    const int blocks = (int)std::min<int64_t>(ceil_div(N * kD, 256), 4 * sm_count());
    CRVQ_CUDA(launch_pdl(hessian_damp_kernel, dim3(blocks), dim3(256), 0, stream, H, N,
                         mem.as<double>(), H_blocks));
    CRVQ_LAUNCHED();
  }
  return CRVQ_OK;
}

crvq_status launch_extract_blocks(const float* H, int64_t N, int d, const int32_t* perm,
                                  float* H_blocks, cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  const int64_t total = (N / d) * d * d;
  const int blocks = (int)std::min<int64_t>(ceil_div(total, 256), 4096);
  ProfScope ps("extract_blocks", stream, (double)total * 8.0);
  CRVQ_CUDA(launch_pdl(extract_blocks_kernel, dim3(blocks), dim3(256), 0, stream, H, N, d, perm,
                       H_blocks, err));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

}  // namespace crvq
