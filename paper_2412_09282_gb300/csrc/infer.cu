// Inference product with a CRVQ-quantized matrix, computed from its codes (the paper's
// inference setting, App. "Inference Speed" / Table speed): Y = X_in W_hat^T, where W_hat in the
// original channel order is the permuted sum of the codebooks' codewords (Sec. 4.3: base
// codebook on every group, extended codebooks on the first G_c groups of the reordered
// channels). W_hat is never formed:
//   y[bi][i] = sum over codebooks s and groups g < G_cov(s) of <C_s[codes_s(i, g)], xs[bi][g]>,
//   xs[bi][p] = X_in[bi][perm[p]]   (the inputs taken once in the sorted channel order).
//
// Layout. A unit is one (codebook, group) pair; a call has U = sum_s G_cov(s) of them. A cluster
// of up to eight CTAs owns a block of rows: each CTA takes a consecutive share of the units for
// all of the block's rows, and the shares meet in distributed shared memory, added in a fixed
// tree: no zeroed counters and no partials in global memory, and results that are identical on every run.
// Two kernels form a share's row sums; both read a row's codes 16 bytes at a time and need no warp
// reduction:
//   table_kernel (one or two inputs, codebooks of up to 1024 / b codewords; a thread per row, one launch,
//     no scratch): the CTA builds the
//     tables lut[unit][k] = <C_s[k], xs[unit]> of 32 units at a time, a code is one entry.
//     Entries are 4 b bytes at random banks, about 3.5 b bank passes per warp and unit.
//   dot_kernel (the rest; after sort_inputs_kernel, which writes the inputs in the sorted order to
//     scratch): a code's codeword is read and dotted with the unit's inputs. With
//     three or more inputs a table entry spans 16-32 bytes, costs as many random bank passes as
//     the codeword itself, and 256 entries are built for the few hundred rows that use them, so
//     tables lose. The codebook is held eight times, copy c in 16-byte bank group c: the eight
//     lanes of a quarter warp read eight different bank groups whatever their codes are, without
//     conflicts. A thread takes four rows, so a unit's inputs are read once for four of them.
//     Codebooks above 512 codewords are read from L2.
//
// What bounds it: the codes are the only per-element stream from memory (4 bytes each); below
// that the shared-memory passes of the lookups (table) and the fp32 FMAs (dot, 8 per input), and in
// both the latency of few warps per SM. Measured (device time per call, K = 256, two extended
// codebooks on 2% of the channels; before: tables built by a kernel of their own, a warp per row
// with a shuffle reduction, partials in global memory):
//   11008 x 4096, one input: 88 -> 16.6 us;  512 x 512, one input: 29 -> 6.4 us;
//   4096 x 11008, eight inputs: 305 -> 49 us.
// Copying the codes to shared memory asynchronously instead of loading them by row was slower
// (21.9 / 8.3 / 65 us), and so were clusters of four for the tables (21.5 us: twice the row
// blocks, so twice the table builds) and of eight for the dots (74 us: 16 clusters where 15 fit).
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace crvq {

namespace {

namespace cg = cooperative_groups;

constexpr int kMaxBatch = 8;
constexpr int kMvCluster = 8;               // CTAs per cluster at most (portable size)
constexpr int kTabCluster = 8;              // table_kernel: few row blocks, so few table builds
constexpr int kDotCluster = 4;              // dot_kernel: more SMs in use (144 of 152)
constexpr int kMvMinRows = 64;              // rows per cluster at least
constexpr int kTabThreads = 768;            // table_kernel: rows (threads) per CTA at most
constexpr int kTabMinThreads = 256;         // table building wants this many threads
constexpr int kTabUnits = 32;               // units whose tables are resident at a time
constexpr int kTabMaxEntries = 1024;        // K * b of a codebook with tables at most
constexpr int kDotThreads = 256;
constexpr int kDotRows = 4;                 // rows per thread
constexpr int kDotCopies = 8;               // one per 16-byte bank group
constexpr int kDotStageK = 512;             // codebooks held in shared memory up to this size
constexpr int kXUnits = 192;                // units whose inputs are resident at a time
// dot_kernel adds a warp's units in runs of eight, or of kDotFold when it has more than 128 of them, and
// then the runs: added one after another, the 268 units of a warp in a 28672 x 8192 product left three
// times the error of a tree. Error against 64 bits (2-norm, three inputs) of a warp-wide tree per 32 units
// / one chain / these runs: 512 x 512 8.5 / 8.9 / 8.5e-8, 4096 x 4096 1.11 / 1.20 / 1.06e-7, 28672 x 8192
// 1.34 / 3.07 / 1.27e-7. The runs and dot8's second chain cost 4% (eight inputs) to 10% (three).
constexpr int kDotFold = 16;

struct MatvecArgs {
  const float* X;       // b x N, row stride ldx
  int64_t ldx;
  int64_t N;
  const int32_t* perm;  // N or null (identity)
  CbList cbs;
  int u_begin[kMaxCodebooks + 1];  // first unit of each codebook
  uint8_t vec[kMaxCodebooks];      // its code rows can be read 16 bytes at a time
  int64_t M;
  int b;
  int units_cta;        // units per CTA share (a multiple of 4)
  int lut_k;            // table stride: the largest K, at least 256 (table_kernel)
  int rows;             // rows per cluster
  int fold;             // units per run of a sum, a power of two (dot_kernel)
  const float* xs;      // [N / 8][BP][8]: the inputs in the sorted order (dot_kernel)
  float* Y;             // b x M, row stride ldy
  int64_t ldy;
};

// Inputs of the units [ua, ue) of codebook s through the permutation:
// xs[(u - ua)][bi][j], zeros for the inputs past b.
template <int BP>
__device__ __forceinline__ void gather_inputs(const MatvecArgs& a, int s, int ua, int ue,
                                              float* xs, unsigned* err) {
  for (int e = threadIdx.x; e < (ue - ua) * kD; e += blockDim.x) {
    int64_t src = (int64_t)(ua - a.u_begin[s]) * kD + e;
    if (a.perm) {
      src = __ldg(a.perm + src);
      if (src < 0 || src >= a.N) {
        raise_error(err, ERRBIT_INDEX);
        src = -1;
      }
    }
#pragma unroll
    for (int bi = 0; bi < BP; ++bi)
      xs[((e >> 3) * BP + bi) * kD + (e & 7)] =
          (src >= 0 && bi < a.b) ? __ldg(a.X + bi * a.ldx + src) : 0.f;
  }
}

// The inputs in the sorted channel order, out[g][bi][j] (zeros for bi >= b), once per call: a
// scattered read per value, which every row block of dot_kernel would otherwise repeat.
template <int BP>
__global__ void __launch_bounds__(256)
sort_inputs_kernel(const float* __restrict__ X, int64_t ldx, int64_t N,
                   const int32_t* __restrict__ perm, int b, float* __restrict__ out,
                   unsigned* err) {
  pdl_trigger();
  pdl_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N) return;
  int64_t src = e;
  if (perm) {
    src = __ldg(perm + e);
    if (src < 0 || src >= N) {
      raise_error(err, ERRBIT_INDEX);
      src = -1;
    }
  }
#pragma unroll
  for (int bi = 0; bi < BP; ++bi)
    out[((e >> 3) * BP + bi) * kD + (e & 7)] = (src >= 0 && bi < b) ? __ldg(X + bi * ldx + src) : 0.f;
}

// <c, x>, two 4-term FMA chains (a single chain of eight rounds more; see kDotFold).
__device__ __forceinline__ float dot8(const float4& c0, const float4& c1, const float4& x0,
                                      const float4& x1) {
  float v = c0.x * x0.x, w = c1.x * x1.x;
  v = fmaf(c0.y, x0.y, v);
  w = fmaf(c1.y, x1.y, w);
  v = fmaf(c0.z, x0.z, v);
  w = fmaf(c1.z, x1.z, w);
  return fmaf(c0.w, x0.w, v) + fmaf(c1.w, x1.w, w);
}

// Y of this cluster's rows from its CTAs' shares part[row][BP] in distributed shared memory, in a
// fixed tree; the CTAs split the rows. Synchronizes the cluster before and after.
template <int BP>
__device__ __forceinline__ void cluster_rows(const MatvecArgs& a, float* part, int64_t r0, int nr) {
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), csize = (int)cluster.num_blocks();
  const int nt = blockDim.x;
  cluster.sync();
  for (int e = rank * nt + (int)threadIdx.x; e < nr * a.b; e += csize * nt) {
    const int bi = e / nr, r = e - bi * nr;
    float v[kMvCluster];
#pragma unroll
    for (int c = 0; c < kMvCluster; ++c)
      v[c] = c < csize ? cluster.map_shared_rank(part, c)[r * BP + bi] : 0.f;
#pragma unroll
    for (int h = kMvCluster / 2; h > 0; h >>= 1)
#pragma unroll
      for (int c = 0; c < h; ++c) v[c] += v[c + h];
    a.Y[bi * a.ldy + r0 + r] = v[0];
  }
  cluster.sync();  // no CTA leaves while its shared memory may still be read
}

// One or two inputs, tables. A thread per row (rows <= blockDim.x); K256: every codebook has at
// most 256 codewords and the table stride is the constant 256.
template <int BP, bool K256>
__global__ void __launch_bounds__(kTabThreads)
table_kernel(const __grid_constant__ MatvecArgs a, int units_sub, unsigned* err) {
  extern __shared__ __align__(16) float sm[];
  float* part = sm;                                // [rows][BP]
  float* xs = part + (size_t)a.rows * BP;          // [kXUnits][BP][8]
  float* lut = xs + kXUnits * BP * kD;             // [units_sub][lut_k][BP]
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), csize = (int)cluster.num_blocks();
  const int64_t r0 = (int64_t)(blockIdx.x / csize) * a.rows;
  const int nr = (int)min((int64_t)a.rows, a.M - r0);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int U = a.u_begin[a.cbs.n];
  const int u0 = min(U, rank * a.units_cta), u1 = min(U, u0 + a.units_cta);
  const int stride = (K256 ? 256 : a.lut_k) * BP;
  const bool live = tid < nr;
  const int64_t i = r0 + (live ? tid : 0);
  float acc[BP];
#pragma unroll
  for (int bi = 0; bi < BP; ++bi) acc[bi] = 0.f;

  for (int s = 0; s < a.cbs.n; ++s) {
    const int ra = max(u0, a.u_begin[s]), re = min(u1, a.u_begin[s + 1]);
    if (ra >= re) continue;
    const CbView& cb = a.cbs.cb[s];
    const int K = cb.K;
    const int32_t* codes = cb.codes + i * cb.ld - a.u_begin[s];  // codes[u]
    // 16-byte loads: aligned rows, and the run starts at a multiple of four groups
    const bool vec = a.vec[s] && ((ra - a.u_begin[s]) & 3) == 0;
    for (int xa = ra; xa < re; xa += kXUnits) {
      const int xe = min(re, xa + kXUnits);
      __syncthreads();  // the previous inputs and tables have been read
      gather_inputs<BP>(a, s, xa, xe, xs, err);
      for (int ua = xa; ua < xe; ua += units_sub) {
        const int n = min(units_sub, xe - ua);
        // this row's codes of the units, in flight while the tables are built
        int32_t k[kTabUnits];
#pragma unroll
        for (int w = 0; w < kTabUnits / 4; ++w) {
          if (vec && 4 * w + 4 <= n) {
            const int4 q = __ldg(reinterpret_cast<const int4*>(codes + ua) + w);
            k[4 * w] = q.x;
            k[4 * w + 1] = q.y;
            k[4 * w + 2] = q.z;
            k[4 * w + 3] = q.w;
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              k[4 * w + e] = 4 * w + e < n ? __ldg(codes + ua + 4 * w + e) : 0;
          }
        }
        __syncthreads();  // inputs written; the previous tables read
        // a thread takes a codeword and walks its thread group's units
        const int kt = min(nt, (K + 31) & ~31), ng = nt / kt, grp = tid / kt;
        if (grp < ng)
          for (int kk = tid - grp * kt; kk < K; kk += kt) {
            const float4 c0 = __ldg(reinterpret_cast<const float4*>(cb.C + (int64_t)kk * kD));
            const float4 c1 = __ldg(reinterpret_cast<const float4*>(cb.C + (int64_t)kk * kD + 4));
#pragma unroll 4
            for (int u = grp; u < n; u += ng) {
              const float* x = xs + (size_t)(ua - xa + u) * BP * kD;
#pragma unroll
              for (int bi = 0; bi < BP; ++bi)
                lut[u * stride + kk * BP + bi] =
                    dot8(c0, c1, *reinterpret_cast<const float4*>(x + bi * kD),
                         *reinterpret_cast<const float4*>(x + bi * kD + 4));
            }
          }
        __syncthreads();
        if (live) {
          // one test for all codes of the batch; a bad code is then skipped and reported
          uint32_t worst = 0;
#pragma unroll
          for (int w = 0; w < kTabUnits; ++w)
            if (w < n) worst = max(worst, (uint32_t)k[w]);
          const bool bad = worst >= (uint32_t)K;
          if (bad) raise_error(err, ERRBIT_INDEX);
          float t[kTabUnits / 4][BP];  // sums of four units, then a balanced tree
          auto lookup = [&](auto clean) {  // clean: whole groups of four units, every code good
#pragma unroll
            for (int w = 0; w < kTabUnits / 4; ++w) {
#pragma unroll
              for (int bi = 0; bi < BP; ++bi) t[w][bi] = 0.f;
              if (4 * w < n) {
                float v[4][BP];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const int u = 4 * w + e;
                  const bool in = clean || (u < n && (uint32_t)k[u] < (uint32_t)K);
                  const float* p = lut + u * stride + (in ? k[u] : 0) * BP;
                  if constexpr (BP == 2) {
                    const float2 q = *reinterpret_cast<const float2*>(p);
                    v[e][0] = in ? q.x : 0.f;
                    v[e][1] = in ? q.y : 0.f;
                  } else {
                    v[e][0] = in ? *p : 0.f;
                  }
                }
#pragma unroll
                for (int bi = 0; bi < BP; ++bi)
                  t[w][bi] = (v[0][bi] + v[1][bi]) + (v[2][bi] + v[3][bi]);
              }
            }
          };
          if (!bad && (n & 3) == 0)
            lookup(std::true_type{});
          else
            lookup(std::false_type{});
#pragma unroll
          for (int h = kTabUnits / 8; h > 0; h >>= 1)
#pragma unroll
            for (int w = 0; w < h; ++w)
#pragma unroll
              for (int bi = 0; bi < BP; ++bi) t[w][bi] += t[w + h][bi];
#pragma unroll
          for (int bi = 0; bi < BP; ++bi) acc[bi] += t[0][bi];
        }
      }
    }
  }
  if (tid < a.rows)
#pragma unroll
    for (int bi = 0; bi < BP; ++bi) part[tid * BP + bi] = acc[bi];
  cluster_rows<BP>(a, part, r0, nr);
}

// Any number of inputs, codewords dotted. A warp takes 32 kDotRows rows (lane l rows l, l + 32,
// ...); a CTA has warps_r warps along the rows and the rest along its share of the units.
template <int BP>
__global__ void __launch_bounds__(kDotThreads, BP == 8 ? 1 : 2)
dot_kernel(const __grid_constant__ MatvecArgs a, int warps_r, unsigned* err) {
  pdl_wait();  // the sorted inputs; the kernels before them may have written codes or codewords
  extern __shared__ __align__(16) float sm[];
  float* part = sm;                                 // [rows][BP]
  float* xs = part + (size_t)a.rows * BP;           // [kXUnits][BP][8]
  float4* cws = reinterpret_cast<float4*>(xs + kXUnits * BP * kD);  // [2][K][kDotCopies]
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), csize = (int)cluster.num_blocks();
  const int64_t r0 = (int64_t)(blockIdx.x / csize) * a.rows;
  const int nr = (int)min((int64_t)a.rows, a.M - r0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wr = warp % warps_r, wu = warp / warps_r, nwu = (kDotThreads / 32) / warps_r;
  const int U = a.u_begin[a.cbs.n];
  const int u0 = min(U, rank * a.units_cta), u1 = min(U, u0 + a.units_cta);
  const int row0 = wr * 32 * kDotRows + lane;       // this lane's first row in the block
  // the sums of the present run of units, and of the runs before it
  float acc[kDotRows][BP], tot[kDotRows][BP];
#pragma unroll
  for (int q = 0; q < kDotRows; ++q)
#pragma unroll
    for (int bi = 0; bi < BP; ++bi) acc[q][bi] = tot[q][bi] = 0.f;
  auto fold = [&]() {
#pragma unroll
    for (int q = 0; q < kDotRows; ++q)
#pragma unroll
      for (int bi = 0; bi < BP; ++bi) {
        tot[q][bi] += acc[q][bi];
        acc[q][bi] = 0.f;
      }
  };

  for (int s = 0; s < a.cbs.n; ++s) {
    const int ra = max(u0, a.u_begin[s]), re = min(u1, a.u_begin[s + 1]);
    if (ra >= re) continue;
    const CbView& cb = a.cbs.cb[s];
    const int K = cb.K;
    const bool staged = K <= kDotStageK;
    const bool vec = a.vec[s] && ((ra - a.u_begin[s]) & 3) == 0;
    const int32_t* codes[kDotRows];  // codes[q][u]; rows past the block repeat its last one
#pragma unroll
    for (int q = 0; q < kDotRows; ++q)
      codes[q] = cb.codes + (r0 + min(row0 + 32 * q, nr - 1)) * cb.ld - a.u_begin[s];
    for (int xa = ra; xa < re; xa += kXUnits) {
      const int xe = min(re, xa + kXUnits);
      __syncthreads();  // the previous inputs and codewords have been read
      if (staged && xa == ra)
        for (int e = tid; e < K * kDotCopies; e += kDotThreads) {
          const float4* c = reinterpret_cast<const float4*>(cb.C + (int64_t)(e / kDotCopies) * kD);
          cws[e] = __ldg(c);
          cws[K * kDotCopies + e] = __ldg(c + 1);
        }
      {
        const float4* src = reinterpret_cast<const float4*>(a.xs) + (size_t)(xa - a.u_begin[s]) * BP * 2;
        for (int e = tid; e < (xe - xa) * BP * 2; e += kDotThreads)
          reinterpret_cast<float4*>(xs)[e] = __ldcg(src + e);
      }
      __syncthreads();
      // this warp's units, a multiple of four
      const int per = ((xe - xa + 4 * nwu - 1) / (4 * nwu)) * 4;
      const int wa = min(xe, xa + wu * per), we = min(xe, wa + per);
      if (wr * 32 * kDotRows >= nr) continue;  // whole warps without rows
      auto load4 = [&](int ua, int32_t k[kDotRows][4]) {  // codes of the units ua .. ua + 3
#pragma unroll
        for (int q = 0; q < kDotRows; ++q) {
          if (vec && ua + 4 <= we) {
            const int4 c = __ldg(reinterpret_cast<const int4*>(codes[q] + ua));
            k[q][0] = c.x;
            k[q][1] = c.y;
            k[q][2] = c.z;
            k[q][3] = c.w;
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) k[q][e] = ua + e < we ? __ldg(codes[q] + ua + e) : 0;
          }
        }
      };
      int32_t kn[kDotRows][4];
      if (wa < we) load4(wa, kn);
      for (int ua = wa; ua < we; ua += 4) {
        int32_t k[kDotRows][4];
#pragma unroll
        for (int q = 0; q < kDotRows; ++q)
#pragma unroll
          for (int e = 0; e < 4; ++e) k[q][e] = kn[q][e];
        if (ua + 4 < we) load4(ua + 4, kn);  // the next four, in flight meanwhile
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (ua + e >= we) break;
          float4 c0[kDotRows], c1[kDotRows];
#pragma unroll
          for (int q = 0; q < kDotRows; ++q) {
            const int32_t kk = k[q][e];
            const bool ok = (uint32_t)kk < (uint32_t)K;
            if (!ok) raise_error(err, ERRBIT_INDEX);
            if (staged) {
              const int at = (ok ? kk : 0) * kDotCopies + (lane & (kDotCopies - 1));
              c0[q] = cws[at];
              c1[q] = cws[K * kDotCopies + at];
            } else {
              const float4* c = reinterpret_cast<const float4*>(cb.C + (int64_t)(ok ? kk : 0) * kD);
              c0[q] = __ldg(c);
              c1[q] = __ldg(c + 1);
            }
            if (!ok) c0[q] = c1[q] = make_float4(0.f, 0.f, 0.f, 0.f);
          }
          const float4* x = reinterpret_cast<const float4*>(xs + (size_t)(ua + e - xa) * BP * kD);
#pragma unroll
          for (int bi = 0; bi < BP; ++bi) {
            const float4 x0 = x[2 * bi], x1 = x[2 * bi + 1];
#pragma unroll
            for (int q = 0; q < kDotRows; ++q) acc[q][bi] += dot8(c0[q], c1[q], x0, x1);
          }
        }
        if (((ua - wa) & (a.fold - 1)) == a.fold - 4) fold();
      }
      fold();
    }
  }
  // the warps along the units add their sums one after another
  for (int w = 0; w < nwu; ++w) {
    if (wu == w)
#pragma unroll
      for (int q = 0; q < kDotRows; ++q) {
        float* p = part + (row0 + 32 * q) * BP;
#pragma unroll
        for (int bi = 0; bi < BP; ++bi) p[bi] = w == 0 ? tot[q][bi] : p[bi] + tot[q][bi];
      }
    __syncthreads();
  }
  cluster_rows<BP>(a, part, r0, nr);
}

template <class Kernel>
crvq_status launch_clusters(Kernel kernel, const MatvecArgs& a, int csize, int threads, size_t smem,
                            bool pdl, int extra, unsigned* err, cudaStream_t stream) {
  CRVQ_TRY(smem_limit((const void*)kernel, smem));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ceil_div(a.M, a.rows) * csize));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  CRVQ_CUDA(cudaLaunchKernelEx(&cfg, kernel, a, extra, err));
  CRVQ_LAUNCHED();
  return CRVQ_OK;
}

// Clusters resident at one CTA per SM: 15 clusters of eight fit the 152 SMs
// (cudaOccupancyMaxActiveClusters; a 16th runs as a second wave), 36 of four, 76 of two.
int64_t cluster_slots(int csize) {
  const int64_t n = sm_count();
  return std::max<int64_t>(1, csize >= 8 ? n * 4 / 5 / 8 : (csize == 4 ? n * 18 / 19 / 4 : n / csize));
}

template <int BP>
crvq_status launch_table(MatvecArgs& a, int csize, unsigned* err, cudaStream_t stream) {
  // a row block per cluster slot (as many rows as possible share a table), at most a thread per row
  int64_t rows = ceil_div(a.M, cluster_slots(csize));
  rows = ceil_div(ceil_div(rows, ceil_div(rows, kTabThreads)), 32) * 32;
  rows = std::max<int64_t>(kMvMinRows, rows);
  a.rows = (int)rows;
  const int threads = (int)std::max<int64_t>(kTabMinThreads, rows);
  const bool k256 = a.lut_k <= 256;
  if (k256) a.lut_k = 256;
  const size_t unit_bytes = (size_t)a.lut_k * BP * 4;
  // units per table set: at most 32 and 128 KB, in equal parts of the share
  const int most = (int)std::min<size_t>(kTabUnits, (128 * 1024) / unit_bytes / 4 * 4);
  const int sub = (int)ceil_div(ceil_div(a.units_cta, ceil_div(a.units_cta, most)), 4) * 4;
  const size_t smem = (size_t)rows * BP * 4 + (size_t)kXUnits * BP * kD * 4 + sub * unit_bytes;
  if (k256) return launch_clusters(table_kernel<BP, true>, a, csize, threads, smem, false, sub, err, stream);
  return launch_clusters(table_kernel<BP, false>, a, csize, threads, smem, false, sub, err, stream);
}

template <int BP>
crvq_status launch_dot(MatvecArgs& a, int csize, int stage_k, unsigned* err, cudaStream_t stream) {
  // warps along the rows: enough that the row blocks fill the cluster slots, no more
  constexpr int kWarpRows = 32 * kDotRows;
  const int64_t rows = ceil_div(a.M, cluster_slots(csize));
  int warps_r = 1;
  while (warps_r < kDotThreads / 32 && warps_r * kWarpRows < rows) warps_r *= 2;
  a.rows = warps_r * kWarpRows;
  a.fold = (int64_t)a.units_cta * warps_r <= 128 * (kDotThreads / 32) ? 8 : kDotFold;
  const size_t smem = (size_t)a.rows * BP * 4 + (size_t)kXUnits * BP * kD * 4 +
                      (size_t)stage_k * kDotCopies * kD * 4;
  Scratch mem;
  CRVQ_TRY(mem.alloc((size_t)a.N * BP * sizeof(float), stream));
  a.xs = mem.as<float>();
  CRVQ_CUDA(launch_pdl(sort_inputs_kernel<BP>, dim3((unsigned)ceil_div(a.N, 256)), dim3(256), 0,
                       stream, a.X, a.ldx, a.N, a.perm, a.b, mem.as<float>(), err));
  CRVQ_LAUNCHED();
  return launch_clusters(dot_kernel<BP>, a, csize, kDotThreads, smem, true, warps_r, err, stream);
}

}  // namespace

crvq_status launch_lut_matvec(const float* X, int64_t ldx, int64_t N, int b,
                              const int32_t* perm, const CbList& cbs, int64_t M, float* Y,
                              int64_t ldy, cudaStream_t stream) {
  unsigned* err = nullptr;
  CRVQ_TRY(device_error_word(&err));
  if (b < 1 || b > kMaxBatch)
    return fail(CRVQ_ERR_UNSUPPORTED, "batch of %d inputs: 1 to %d are implemented", b,
                kMaxBatch);
  MatvecArgs a{};
  a.X = X;
  a.ldx = ldx;
  a.N = N;
  a.perm = perm;
  a.cbs = cbs;
  a.M = M;
  a.b = b;
  a.Y = Y;
  a.ldy = ldy;
  int64_t U = 0;
  int stage_k = 0;
  for (int s = 0; s < cbs.n; ++s) {
    const CbView& cb = cbs.cb[s];
    a.u_begin[s] = (int)U;
    U += cb.G_cov;
    a.vec[s] = ((uintptr_t)cb.codes & 15u) == 0 && cb.ld % 4 == 0;
    a.lut_k = std::max(a.lut_k, cb.K);
    if (cb.K <= kDotStageK) stage_k = std::max(stage_k, cb.K);
    if (U > INT32_MAX / 2) return fail(CRVQ_ERR_UNSUPPORTED, "too many (codebook, group) pairs");
  }
  a.u_begin[cbs.n] = (int)U;
  // cluster size: at least four units per CTA; shares of whole multiples of four units, so that
  // a share of the base codebook starts on a 16-byte boundary of its code rows
  const bool tables = b <= 2 && (int64_t)a.lut_k * b <= kTabMaxEntries;
  int csize = tables ? kTabCluster : kDotCluster;
  while (csize > 1 && U < 4 * csize) csize >>= 1;
  a.units_cta = (int)(std::max<int64_t>(1, ceil_div(ceil_div(U, csize), 4)) * 4);
  ProfScope ps("matvec_slices", stream, (double)M * (N / kD) * cbs.n);
  if (tables) return b == 1 ? launch_table<1>(a, csize, err, stream) : launch_table<2>(a, csize, err, stream);
  if (b == 1) return launch_dot<1>(a, csize, stage_k, err, stream);
  if (b == 2) return launch_dot<2>(a, csize, stage_k, err, stream);
  if (b <= 4) return launch_dot<4>(a, csize, stage_k, err, stream);
  return launch_dot<8>(a, csize, stage_k, err, stream);
}

}  // namespace crvq
