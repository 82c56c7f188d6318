// Graph low-pass filter (Eq. 5) and its FSLR selection (Eq. 6, Section 2.4) as
// a kernel of their own (k_filter, the device routine in select.cuh), the
// output of a chosen iterate in input order, and the graph / FSLR exports.
#include <algorithm>
#include <climits>

#include "select.cuh"

namespace fgbd {
namespace {

// NX further neighbour slots per point: 0 at window 1, 6 (w - 1) at window w;
// DEEP: contexts that store more than kSpecSure steps
template <int NX, bool DEEP = false>
__global__ void __launch_bounds__(kFilterThreads, 2) k_filter(FilterArgs a) {
  pdl_wait();
  // the stored steps count only if the noise-estimate launch finished them
  __shared__ int s_S;
  if (threadIdx.x == 0) {
    const int done = int(ld_acquire_u32(reinterpret_cast<const uint32_t*>(&a.sc->spec_done)));
    s_S = (a.mode == 0 && a.spec_depth > 0) ? min(done, a.spec_depth) : 0;
  }
  __syncthreads();
  uint32_t epoch = 0;
  select_filter<kFilterThreads, NX, DEEP>(a, s_S, 0, gridDim.x, &a.sc->barrier, epoch, 2);
}

// Segmented (window 1): frame f's blocks [start[f], start[f + 1]) select and
// filter frame f, with grid barriers among themselves only.
template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) k_filter_seg(const __grid_constant__ Seg<FilterArgs> s) {
  pdl_wait();
  const int f = seg_frame(s, blockIdx.x);
  const FilterArgs& a = s.a[f];
  __shared__ int s_S;
  if (threadIdx.x == 0) {
    const int done = int(ld_acquire_u32(reinterpret_cast<const uint32_t*>(&a.sc->spec_done)));
    s_S = (a.mode == 0 && a.spec_depth > 0) ? min(done, a.spec_depth) : 0;
  }
  __syncthreads();
  uint32_t epoch = 0;
  select_filter<THREADS, 0, false, SearchPart::kCapped>(a, s_S, s.start[f], uint32_t(s.start[f + 1] - s.start[f]),
                                                        &a.sc->barrier, epoch, 1);
}

// The frames whose search that launch left (resume_t), one after another with every block.
__global__ void __launch_bounds__(kFilterThreads, 2) k_filter_rest_seg(const __grid_constant__ Seg<FilterArgs> s) {
  pdl_wait();
  for (int f = 0; f < s.count; ++f) {
    const FilterArgs& a = s.a[f];
    if (a.sc->resume_t == 0) continue;
    __syncthreads();  // the frame before has left the shared scalars
    uint32_t epoch = 0;
    const int S = min(int(a.sc->spec_done), a.spec_depth);
    select_filter<kFilterThreads, 0, false, SearchPart::kRest>(a, S, 0, gridDim.x, &a.sc->barrier_rest, epoch, 2);
  }
}

__global__ void __launch_bounds__(256) k_output(FilterArgs a) {
  pdl_wait();
  output_quads(a, a.sc->kept_buf, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// ---------------------------------------------------------------- export

constexpr int kScanBlock = 1024;

// Exclusive block prefix of v over the kScanBlock threads; *total: the block's sum.
__device__ __forceinline__ int block_prefix(int v, int* total) {
  constexpr int W = kScanBlock / 32;
  __shared__ int s[W];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int in = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= o) in += t;
  }
  if (lane == 31) s[warp] = in;
  __syncthreads();
  int w = s[lane];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, w, o);
    if (lane >= o) w += t;
  }
  const int before = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
  *total = __shfl_sync(0xffffffffu, w, 31);
  return (warp > 0 ? before : 0) + in - v;
}

// CSR row pointers, part 1: the degree of every point (input order) and its prefix
// within the block of kScanBlock points; totals[b]: the block's sum.  NS slots a point.
template <int NS>
__global__ void __launch_bounds__(kScanBlock)
    k_csr_degree(int n, GraphBufs gb, int64_t* __restrict__ row_ptr, int64_t* __restrict__ totals) {
  pdl_wait();
  const int64_t i = int64_t(blockIdx.x) * kScanBlock + threadIdx.x;
  int deg = 0;
  const int k = i < n ? gb.rank12[i].x : -1;
  if (in_range(k, n)) {
    const uint32_t pkk = gb.pk[k];
    const int4 s = gb.c4[k];
#pragma unroll
    for (int j = 0; j < NS; ++j) deg += neighbour_of(j, k, n, pkk, s, gb.cx, gb.cx_stride) >= 0;
  }
  int total;
  const int before = block_prefix(deg, &total);
  if (i <= n) row_ptr[i] = before;
  if (threadIdx.x == 0) totals[blockIdx.x] = total;
}

// Part 2: what the blocks before hold, added up by each block for itself (one
// thread over all of them took 14 us at 300,000 points).  Block 0 also leaves
// 1 / sigma_g^2 behind the totals, so that no thread of the fill divides in float64.
__global__ void __launch_bounds__(kScanBlock)
    k_csr_row_ptr(int n, int64_t* __restrict__ row_ptr, int64_t* totals, const DevScalars* __restrict__ sc) {
  pdl_wait();
  constexpr int W = kScanBlock / 32;
  __shared__ long long s[W];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  long long sum = 0;
  for (int b = threadIdx.x; b < int(blockIdx.x); b += kScanBlock) sum += totals[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) s[warp] = sum;
  __syncthreads();
  sum = s[lane];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const int64_t i = int64_t(blockIdx.x) * kScanBlock + threadIdx.x;
  if (i <= n) row_ptr[i] += sum;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const double sg = sigma_g_of(sc);
    reinterpret_cast<float*>(totals + gridDim.x)[0] = sg > 0.0 ? float(1.0 / (sg * sg)) : 0.f;
  }
}

// Part 3: the rows, each sorted by the neighbours' input indices.  In C1 order, where
// a point's neighbours lie near those of the points beside it (in input order every
// read is a random one), NS slots in registers; an entry's place in its row is the
// number of smaller indices, and the rows go out from shared memory, G lanes a row,
// since they land anywhere: a store of the whole warp touches one or two sectors a
// row, where one entry of every row at a time touched 32.  Bound by random sectors:
// 300,000 points 14.8 us (in input order, rows in local memory, a float64 division a
// thread: 46), row pointers 10.7 (28 in five launches), cold cache.
template <int NS, int G>
__global__ void __launch_bounds__(256)
    k_csr_fill(int n, int bits, GraphBufs gb, const int64_t* __restrict__ row_ptr, const float* __restrict__ inv2_of,
               int32_t* __restrict__ col, float* __restrict__ w, int64_t col_capacity,
               const DevScalars* __restrict__ sc) {
  static_assert(NS <= G && G <= 32, "a lane an entry");
  pdl_wait();
  __shared__ int s_col[256][NS];
  __shared__ float s_w[256][NS];
  const int lane = threadIdx.x & 31, first = threadIdx.x & ~31;
  const float inv2 = *inv2_of;
  const bool pair = gb.node_sig && sc->sigma_mode == kSigmaPair;
  for (int k0 = blockIdx.x * 256 + first; k0 < n; k0 += gridDim.x * 256) {
    const int k = k0 + lane;
    int cnt = 0;
    long long base = 0;
    if (k < n) {
      const int i = gb.perm1[k];
      const uint32_t pkk = gb.pk[k];
      const int4 s = gb.c4[k];
      if (in_range(i, n)) base = row_ptr[i];
      int nb[NS], orig[NS];
#pragma unroll
      for (int j = 0; j < NS; ++j) nb[j] = neighbour_of(j, k, n, pkk, s, gb.cx, gb.cx_stride);
      float wv[NS];
#pragma unroll
      for (int j = 0; j < NS; ++j) {
        orig[j] = INT_MAX;
        wv[j] = 0.f;
        if (nb[j] >= 0) {
          orig[j] = gb.perm1[nb[j]];
          const float d2 = float(sq_dist_c1(pkk, gb.pk[nb[j]], bits));
          if (pair) {
            // the pair reading: w_ij = exp(-d_ij^2 / (sigma_i sigma_j)); 1 where the product is 0
            const float ss = gb.node_sig[k] * gb.node_sig[nb[j]];
            wv[j] = ss > 0.f ? expf(-d2 / ss) : 1.f;
          } else {
            wv[j] = expf(-d2 * inv2);
          }
          ++cnt;
        }
      }
#pragma unroll
      for (int j = 0; j < NS; ++j) {
        int at = 0;
#pragma unroll
        for (int m = 0; m < NS; ++m) at += orig[m] < orig[j];
        if (nb[j] >= 0) {
          s_col[threadIdx.x][at] = orig[j];
          s_w[threadIdx.x][at] = wv[j];
        }
      }
      if (!in_range(i, n) || base < 0 || base + cnt > col_capacity) cnt = 0;
    }
    __syncwarp();
    const int l = lane % G;
#pragma unroll
    for (int r0 = 0; r0 < 32; r0 += 32 / G) {
      const int r = r0 + lane / G;
      const long long b = __shfl_sync(0xffffffffu, base, r);
      const int c = __shfl_sync(0xffffffffu, cnt, r);
      if (l < NS && l < c) {
        col[b + l] = s_col[first + r][l];
        if (w) w[b + l] = s_w[first + r][l];
      }
    }
    __syncwarp();
  }
}

__global__ void k_spread_export(int n, const int2* __restrict__ rank12, const float* __restrict__ spread,
                                const uint8_t* __restrict__ keep8, float* __restrict__ spread_out,
                                uint8_t* __restrict__ keep_out) {
  pdl_wait();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int k = rank12[i].x;
    if (!in_range(k, n)) continue;
    if (spread_out) spread_out[i] = spread[k];
    if (keep_out) keep_out[i] = keep8[k] ? 1 : 0;
  }
}

}  // namespace

int filter_grid(int n, int num_sms, int nx) {
  int per_sm = 0;
  cudaError_t e;
  if (nx == extra_slots(3))
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter<extra_slots(3)>, kFilterThreads, 0);
  else if (nx == extra_slots(2))
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter<extra_slots(2)>, kFilterThreads, 0);
  else {
    int deep = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter<0>, kFilterThreads, 0);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&deep, k_filter<0, true>, kFilterThreads, 0);
    per_sm = std::min(per_sm, deep);
  }
  if (e != cudaSuccess || per_sm < 1) per_sm = 1;
  const int need = std::max(1, (n + kFilterThreads - 1) / kFilterThreads);
  return std::max(1, std::min(need, per_sm * num_sms));
}

cudaError_t launch_filter(const FilterArgs& a, int grid, cudaStream_t stream) {
  if (a.nx == extra_slots(2))
    return launch_kernel(k_filter<extra_slots(2)>, dim3(grid), dim3(kFilterThreads), 0, stream, true, a);
  if (a.nx == extra_slots(3))
    return launch_kernel(k_filter<extra_slots(3)>, dim3(grid), dim3(kFilterThreads), 0, stream, true, a);
  if (a.nx != 0) return cudaErrorInvalidValue;
  if (a.spec_depth > kSpecSure)
    return launch_kernel(k_filter<0, true>, dim3(grid), dim3(kFilterThreads), 0, stream, true, a);
  return launch_kernel(k_filter<0>, dim3(grid), dim3(kFilterThreads), 0, stream, true, a);
}

int filter_seg_max_per_sm(int threads) {
  int per_sm = 0;
  const cudaError_t e =
      threads == 256 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter_seg<256>, 256, 0)
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter_seg<512>, 512, 0);
  if (e != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return 1;
  }
  return per_sm;
}

cudaError_t launch_filter_seg(const FilterArgs* a, int count, int threads, int filter_per_sm, int num_sms,
                              cudaStream_t stream) {
  if (count < 1 || count > kSegMax || (threads != 256 && threads != 512)) return cudaErrorInvalidValue;
  for (int f = 0; f < count; ++f)
    if (a[f].nx != 0) return cudaErrorInvalidValue;
  // every block must be resident (grid barriers): at most the occupancy per SM
  const int per_sm = std::max(1, std::min(filter_per_sm, filter_seg_max_per_sm(threads)));
  const int pool = per_sm * num_sms;
  if (pool < count) return cudaErrorInvalidValue;
  Seg<FilterArgs> sg;
  int blocks[kSegMax];
  double total = 0.0;
  for (int f = 0; f < count; ++f) total += double(std::max(a[f].n, 1));
  int given = 0;
  for (int f = 0; f < count; ++f) {
    sg.a[f] = a[f];
    // in proportion to the points, at least one block, no more than one thread per point
    const int need = std::max(1, (a[f].n + threads - 1) / threads);
    const int left = count - 1 - f;
    int b = int(double(pool) * double(std::max(a[f].n, 1)) / total);
    b = std::max(1, std::min({b, need, pool - given - left}));
    given += b;
    blocks[f] = b;
  }
  const int grid = seg_layout(sg, blocks, count);
  if (threads == 256) return launch_kernel(k_filter_seg<256>, dim3(grid), dim3(256), 0, stream, true, sg);
  return launch_kernel(k_filter_seg<512>, dim3(grid), dim3(512), 0, stream, true, sg);
}

cudaError_t launch_filter_rest_seg(const FilterArgs* a, int count, int num_sms, cudaStream_t stream) {
  if (count < 1 || count > kSegMax) return cudaErrorInvalidValue;
  int per_sm = 0;
  const cudaError_t e =
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter_rest_seg, kFilterThreads, 0);
  if (e != cudaSuccess) return e;
  Seg<FilterArgs> sg;
  for (int f = 0; f < count; ++f) {
    if (a[f].nx != 0) return cudaErrorInvalidValue;
    sg.a[f] = a[f];
  }
  sg.count = count;
  return launch_kernel(k_filter_rest_seg, dim3(std::max(1, per_sm) * num_sms), dim3(kFilterThreads), 0, stream, true, sg);
}

cudaError_t launch_output(const FilterArgs& a, cudaStream_t stream) {
  if (a.n <= 0) return cudaSuccess;
  const int grid = std::min((a.n + 255) / 256, 152 * 16);
  return launch_kernel(k_output, dim3(grid), dim3(256), 0, stream, false, a);
}

cudaError_t launch_csr_row_ptr(int n, const GraphBufs& gb, int64_t* row_ptr, int64_t* block_tmp,
                               const DevScalars* sc, cudaStream_t stream) {
  const int nb = int((int64_t(n) + 1 + kScanBlock - 1) / kScanBlock);
  const auto degree = gb.nx == extra_slots(3)   ? k_csr_degree<6 + extra_slots(3)>
                      : gb.nx == extra_slots(2) ? k_csr_degree<6 + extra_slots(2)>
                                                : k_csr_degree<6>;
  const cudaError_t e = launch_kernel(degree, dim3(nb), dim3(kScanBlock), 0, stream, false, n, gb, row_ptr, block_tmp);
  if (e != cudaSuccess) return e;
  return launch_kernel(k_csr_row_ptr, dim3(nb), dim3(kScanBlock), 0, stream, false, n, row_ptr, block_tmp, sc);
}

cudaError_t launch_csr_fill(int n, int bits, const GraphBufs& gb, const int64_t* row_ptr, const int64_t* block_tmp,
                            int32_t* col, float* w, int64_t col_capacity, const DevScalars* sc, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int nb = int((int64_t(n) + 1 + kScanBlock - 1) / kScanBlock);
  const float* inv2 = reinterpret_cast<const float*>(block_tmp + nb);
  const int grid = std::min((n + 255) / 256, 152 * 16);
  const auto fill = gb.nx == extra_slots(3)   ? k_csr_fill<6 + extra_slots(3), 32>
                    : gb.nx == extra_slots(2) ? k_csr_fill<6 + extra_slots(2), 16>
                                              : k_csr_fill<6, 8>;
  return launch_kernel(fill, dim3(grid), dim3(256), 0, stream, false, n, bits, gb, row_ptr, inv2, col, w,
                       col_capacity, sc);
}

cudaError_t launch_spread_export(int n, const int2* rank12, const float* spread, const uint8_t* keep8,
                                 float* spread_out, uint8_t* keep_out, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int grid = std::min((n + 255) / 256, 152 * 16);
  return launch_kernel(k_spread_export, dim3(grid), dim3(256), 0, stream, false, n, rank12, spread, keep8, spread_out,
                       keep_out);
}

}  // namespace fgbd
