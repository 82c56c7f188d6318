// Differentiable graph filter: Eq. 5 generalised to a filter strength alpha
// and a weight bandwidth sigma, with its adjoint.
//
//   x_{t+1} = (1 - alpha) x_t + alpha R x_t,   R = D^{-1} W,
//   W_ij = exp(-d_ij^2 / sigma^2) over the scan-line graph (Eq. 4),
// so alpha = 1/2 and sigma = sigma_g give Eq. 5 (W_g = D + W, D_g = 2D).  For a
// loss L(x_q) with g = dL/dx_q and u_t = dL/dx_t:
//   u_t = P^T u_{t+1} = (1 - alpha) u_{t+1} + alpha W D^{-1} u_{t+1}
//   dL/dalpha = sum_t u_{t+1} . (R x_t - x_t)
//   dL/dsigma = sum_t alpha u_{t+1} . (dR/dsigma) x_t,
//   (dR/dsigma x)_i = (2 / sigma^3) sum_j R_ij (d_ij^2 - e_i) x_j,
//   e_i = sum_j R_ij d_ij^2
// (the derivative of a row-normalised Gaussian row; the row-minimum shift
// used against underflow cancels in it).  The rows of R and, for the
// adjoint, the weight of i in each neighbour's row (R^T) are tabulated once
// per forward call.  Iterates are kept every `checkpoint` steps and the ones
// in between are recomputed segment by segment in the backward call.
// Reductions are float64 per block, summed in a fixed order: deterministic.
#include <algorithm>
#include <climits>

#include "fgbd_internal.cuh"

namespace fgbd {
namespace {

constexpr int kDiffThreads = 256;

__device__ __forceinline__ double diff_sigma(double sigma, const DevScalars* sc) {
  return sigma > 0.0 ? sigma : sigma_g_of(sc);
}

// exponent scale of Eq. 4 in powers of two
__host__ __device__ inline float diff_cexp(double sg) {
  return sg > 0.0 ? float(1.4426950408889634 / (sg * sg)) : 0.f;
}
// alpha * 2 / sigma^3, the factor of dL/dsigma
__host__ __device__ inline double diff_dscale(float alpha, double sg) {
  return sg > 0.0 ? double(alpha) * (2.0 / (sg * sg * sg)) : 0.0;
}

// A point's row: the C1 neighbours i - 1 and i + 1 and the four C2/C3 slots, in
// this order everywhere.  The tables hold one value a slot as a float2 (C1) and a
// float4 (C2/C3), so a warp reads whole 128-byte lines of each; the indices are
// the graph's own (24-byte rows, one table for the indices too, made every load
// of a warp touch six lines: at 300,000 points a backward step took 24 us, now
// 14.5; a forward step 8, now 7.4, both with a cold cache).  A slot without a neighbour has R = -1; the one neighbour of a point
// without any is the point itself, in slot 2, whose index is out of range.
struct DiffRow {
  int j[kK];
  float r[kK];
};
__device__ __forceinline__ DiffRow diff_row(int i, int n, const int4* __restrict__ c4, const float2* __restrict__ r2,
                                            const float4* __restrict__ r4) {
  const int4 c = c4[i];
  const float2 a = r2[i];
  const float4 b = r4[i];
  return {{i - 1, i + 1, in_range(c.x, n) ? c.x : i, in_range(c.y, n) ? c.y : i, in_range(c.z, n) ? c.z : i,
           in_range(c.w, n) ? c.w : i},
          {a.x, a.y, b.x, b.y, b.z, b.w}};
}
// (a NaN weight, of a bandwidth whose square underflows, counts as a neighbour)
__device__ __forceinline__ bool diff_linked(float r) { return !(r < 0.f); }

__device__ __forceinline__ float4 diff_colour(const float* __restrict__ rgb, int i, int n) {
  if (!in_range(i, n)) return make_float4(0.f, 0.f, 0.f, 0.f);
  return make_float4(rgb[3 * size_t(i)], rgb[3 * size_t(i) + 1], rgb[3 * size_t(i) + 2], 0.f);
}
__device__ __forceinline__ void diff_put(float* __restrict__ rgb, int i, int n, float4 v) {
  if (!in_range(i, n)) return;
  rgb[3 * size_t(i)] = v.x;
  rgb[3 * size_t(i) + 1] = v.y;
  rgb[3 * size_t(i) + 2] = v.z;
}

// Rows of R, what a neighbour needs to form its weight in this row (rec: packed
// code, smallest squared distance, 1 / sum of weights), and the colours taken into
// the sorted order (x[k] = rgb[perm1[k]]), whose random reads run beside the rows'.
// Bound by those reads: 8.9 us at 300,000 points; as two launches 23 (a float64
// division in every block went before the reads) and 5.3.
__global__ void __launch_bounds__(kDiffThreads)
    k_diff_rows(int n, int bits, double sigma_in, float cexp_in, const uint32_t* __restrict__ pk,
                const int4* __restrict__ c4, const int32_t* __restrict__ perm1, const float* __restrict__ rgb,
                const DevScalars* __restrict__ sc, DiffBufs db, float4* __restrict__ x) {
  pdl_wait();
  __shared__ float s_cexp;
  float cexp = cexp_in;
  if (!(sigma_in > 0.0)) {
    // sigma_g: the exponent scale once per block (float64 is slow on this GPU)
    if (threadIdx.x == 0) s_cexp = diff_cexp(diff_sigma(sigma_in, sc));
    __syncthreads();
    cexp = s_cexp;
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t ci = pk[i];  // packed code, with the same-line variant's missing-C1-link bits
    const int4 s = c4[i];
    const int src = perm1[i];
    const int j[kK] = {c1_prev_linked(ci, i) ? i - 1 : -1,    c1_next_linked(ci, i, n) ? i + 1 : -1,
                       in_range(s.x, n) ? s.x : -1, in_range(s.y, n) ? s.y : -1,
                       in_range(s.z, n) ? s.z : -1, in_range(s.w, n) ? s.w : -1};
    int d2[kK];
    int dmin = INT_MAX;
#pragma unroll
    for (int t = 0; t < kK; ++t) {
      d2[t] = j[t] >= 0 ? sq_dist_c1(ci, pk[j[t]], bits) : INT_MAX;
      dmin = min(dmin, d2[t]);
    }
    const float4 v = diff_colour(rgb, src, n);
    float w[kK];
    float sw = 0.f;
#pragma unroll
    for (int t = 0; t < kK; ++t) {
      w[t] = j[t] >= 0 ? exp2f(float(dmin - d2[t]) * cexp) : 0.f;
      sw += w[t];
    }
    float r[kK];
    const float inv = 1.f / sw;
#pragma unroll
    for (int t = 0; t < kK; ++t) r[t] = j[t] >= 0 ? w[t] * inv : -1.f;
    // no neighbour (a one-point graph): R x = x, as Eq. 5 leaves such a point unchanged
    if (sw == 0.f) r[2] = 1.f;
    db.r2[i] = make_float2(r[0], r[1]);
    db.r4[i] = make_float4(r[2], r[3], r[4], r[5]);
    db.rec[i] = make_int4(int(ci), dmin, __float_as_int(inv), 0);
    x[i] = v;
  }
}

// For the adjoint, per slot: RT, the weight of i in its neighbour's row (the graph
// is symmetric; formed as that row's thread formed it, so with the same bits: one
// 16-byte read a neighbour instead of a search of its row), and G = R_ij (d_ij^2 -
// e_i); and the output's gradient taken into the sorted order.  11.4 us at 300,000
// points; the search took 18, in every forward call, and the gradient's launch 5.3.
__global__ void __launch_bounds__(kDiffThreads)
    k_diff_rows_t(int n, int bits, double sigma_in, float cexp_in, const int4* __restrict__ c4,
                  const int32_t* __restrict__ perm1, const float* __restrict__ grad,
                  const DevScalars* __restrict__ sc, DiffBufs db, float4* __restrict__ u) {
  pdl_wait();
  __shared__ float s_cexp;
  float cexp = cexp_in;
  if (!(sigma_in > 0.0)) {
    if (threadIdx.x == 0) s_cexp = diff_cexp(diff_sigma(sigma_in, sc));
    __syncthreads();
    cexp = s_cexp;
  }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const DiffRow row = diff_row(i, n, c4, db.r2, db.r4);
    const uint32_t ci = uint32_t(db.rec[i].x);
    const int src = perm1[i];
    int4 nb[kK];
#pragma unroll
    for (int t = 0; t < kK; ++t)
      nb[t] = diff_linked(row.r[t]) ? db.rec[row.j[t]] : make_int4(0, 0, 0, 0);
    const float4 v = diff_colour(grad, src, n);
    float rt[kK], d2[kK];
    float ei = 0.f;
#pragma unroll
    for (int t = 0; t < kK; ++t) {
      rt[t] = d2[t] = 0.f;
      if (diff_linked(row.r[t])) {
        if (row.j[t] == i) {
          rt[t] = row.r[t];
        } else {
          const int d = sq_dist_c1(ci, uint32_t(nb[t].x), bits);
          d2[t] = float(d);
          rt[t] = exp2f(float(nb[t].y - d) * cexp) * __int_as_float(nb[t].z);
        }
        ei = fmaf(row.r[t], d2[t], ei);
      }
    }
    float g[kK];
#pragma unroll
    for (int t = 0; t < kK; ++t) g[t] = row.r[t] * (d2[t] - ei);
    db.rt2[i] = make_float2(rt[0], rt[1]);
    db.rt4[i] = make_float4(rt[2], rt[3], rt[4], rt[5]);
    db.g2[i] = make_float2(g[0], g[1]);
    db.g4[i] = make_float4(g[2], g[3], g[4], g[5]);
    u[i] = v;
  }
}

// out[perm1[k]] = x[k] (sorted order -> input order), where no step writes it
__global__ void __launch_bounds__(kDiffThreads)
    k_diff_scatter(int n, const float4* __restrict__ x, const int32_t* __restrict__ perm1, float* __restrict__ out) {
  pdl_wait();
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
    diff_put(out, perm1[k], n, x[k]);
}

// One forward step: dst = (1 - alpha) src + alpha R src.  The last one writes the
// result in input order (out) instead.  Bound by the neighbours' reads.
template <bool LAST>
__global__ void __launch_bounds__(kDiffThreads)
    k_diff_step(int n, float alpha, const int4* __restrict__ c4, const float2* __restrict__ r2,
                const float4* __restrict__ r4, const float4* __restrict__ src, float4* __restrict__ dst,
                const int32_t* __restrict__ perm1, float* __restrict__ out) {
  pdl_wait();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const DiffRow row = diff_row(i, n, c4, r2, r4);
    const float4 s = src[i];
    const int to = LAST ? perm1[i] : 0;
    float rx = 0.f, ry = 0.f, rz = 0.f;
#pragma unroll
    for (int t = 0; t < kK; ++t) {
      if (diff_linked(row.r[t])) {
        const float4 v = src[row.j[t]];
        rx = fmaf(row.r[t], v.x, rx);
        ry = fmaf(row.r[t], v.y, ry);
        rz = fmaf(row.r[t], v.z, rz);
      }
    }
    const float a = 1.f - alpha;
    const float4 o = make_float4(fmaf(a, s.x, alpha * rx), fmaf(a, s.y, alpha * ry), fmaf(a, s.z, alpha * rz), 0.f);
    if constexpr (LAST) diff_put(out, to, n, o);
    else dst[i] = o;
  }
}

// Float-float accumulator (hi + lo): TwoSum (Knuth) and the TwoProduct of a
// fused multiply-add keep products and sums of float32 values exact to about
// 44 bits without float64, which is slow on this GPU.
struct FF2 {
  float hi, lo;
};
__device__ __forceinline__ FF2 ff2_add(FF2 x, FF2 y) {
  const float s = __fadd_rn(x.hi, y.hi);
  const float bb = __fsub_rn(s, x.hi);
  const float err = __fadd_rn(__fsub_rn(x.hi, __fsub_rn(s, bb)), __fsub_rn(y.hi, bb));
  const float lo = __fadd_rn(err, __fadd_rn(x.lo, y.lo));
  const float h = __fadd_rn(s, lo);
  return {h, __fsub_rn(lo, __fsub_rn(h, s))};
}
// x += a * b, the product exact
__device__ __forceinline__ FF2 ff2_fma(FF2 x, float a, float b) {
  const float p = __fmul_rn(a, b);
  return ff2_add(x, {p, fmaf(a, b, -p)});
}
__device__ __forceinline__ FF2 ff2_shfl_down(FF2 x, int o) {
  return {__shfl_down_sync(0xffffffffu, x.hi, o), __shfl_down_sync(0xffffffffu, x.lo, o)};
}

// One adjoint step: u_out = P^T u (the last one, t = 0, writes it in input order
// to grad_in instead), and this step's terms of dL/dalpha and dL/dsigma (without
// its factor), added to the block's float64 pair partial[blockIdx.x] (`first`: the
// pair is set).  The per-point terms are accumulated in float-float and only the
// block's warp sums are combined in float64, as a tree: a chain of sixteen float64
// additions in one thread, and the factor's division in every block, had cost
// as much as the reads.
template <bool LAST>
__global__ void __launch_bounds__(kDiffThreads)
    k_diff_back_step(int n, float alpha, bool first, const int4* __restrict__ c4, DiffBufs db,
                     const float4* __restrict__ x, const float4* __restrict__ u, float4* __restrict__ u_out,
                     const int32_t* __restrict__ perm1, float* __restrict__ grad_in, double2* __restrict__ partial) {
  pdl_wait();
  constexpr int W = kDiffThreads / 32;
  __shared__ FF2 s_red[2][W];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double2 before = make_double2(0.0, 0.0);
  if (threadIdx.x == 0 && !first) before = partial[blockIdx.x];
  FF2 da = {0.f, 0.f}, ds = {0.f, 0.f};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const DiffRow row = diff_row(i, n, c4, db.r2, db.r4);
    const float2 ta = db.rt2[i], ga = db.g2[i];
    const float4 tb = db.rt4[i], gb = db.g4[i];
    const float rt[kK] = {ta.x, ta.y, tb.x, tb.y, tb.z, tb.w}, gg[kK] = {ga.x, ga.y, gb.x, gb.y, gb.z, gb.w};
    const float4 ui = u[i];
    const float4 xi = x[i];
    const int to = LAST ? perm1[i] : 0;
    float ux = 0.f, uy = 0.f, uz = 0.f;  // (W D^-1 u)_i
    float rx = 0.f, ry = 0.f, rz = 0.f;  // (R x)_i
    float gx = 0.f, gy = 0.f, gz = 0.f;  // sum_j R_ij (d2_ij - e_i) x_j
#pragma unroll
    for (int t = 0; t < kK; ++t) {
      if (diff_linked(row.r[t])) {
        const float4 uj = u[row.j[t]];
        const float4 xj = x[row.j[t]];
        ux = fmaf(rt[t], uj.x, ux);
        uy = fmaf(rt[t], uj.y, uy);
        uz = fmaf(rt[t], uj.z, uz);
        rx = fmaf(row.r[t], xj.x, rx);
        ry = fmaf(row.r[t], xj.y, ry);
        rz = fmaf(row.r[t], xj.z, rz);
        gx = fmaf(gg[t], xj.x, gx);
        gy = fmaf(gg[t], xj.y, gy);
        gz = fmaf(gg[t], xj.z, gz);
      }
    }
    const float a = 1.f - alpha;
    const float4 o = make_float4(fmaf(a, ui.x, alpha * ux), fmaf(a, ui.y, alpha * uy), fmaf(a, ui.z, alpha * uz), 0.f);
    if constexpr (LAST) diff_put(grad_in, to, n, o);
    else u_out[i] = o;
    da = ff2_fma(ff2_fma(ff2_fma(da, ui.x, rx - xi.x), ui.y, ry - xi.y), ui.z, rz - xi.z);
    ds = ff2_fma(ff2_fma(ff2_fma(ds, ui.x, gx), ui.y, gy), ui.z, gz);
  }
  // block sums in a fixed order
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    da = ff2_add(da, ff2_shfl_down(da, o));
    ds = ff2_add(ds, ff2_shfl_down(ds, o));
  }
  if (lane == 0) {
    s_red[0][warp] = da;
    s_red[1][warp] = ds;
  }
  __syncthreads();
  if (warp == 0) {
    static_assert(2 * W <= 32, "a lane a warp sum");
    const FF2 v = lane < 2 * W ? s_red[lane / W][lane % W] : FF2{0.f, 0.f};
    double sum = double(v.hi) + double(v.lo);
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o, W);
    const double sig = __shfl_sync(0xffffffffu, sum, W);
    if (lane == 0) partial[blockIdx.x] = make_double2(before.x + sum, before.y + sig);
  }
}

constexpr int kDiffReduceThreads = 1024;

// grad[0..1] = the sums of the blocks' (dalpha, dsigma) pairs, in a fixed order, the
// second times alpha 2 / sigma^3
__global__ void __launch_bounds__(kDiffReduceThreads)
    k_diff_reduce(int count, float alpha, double sigma_in, double scale_in, const DevScalars* __restrict__ sc,
                  const double2* __restrict__ partial, double* __restrict__ grad) {
  pdl_wait();
  constexpr int W = kDiffReduceThreads / 32;
  __shared__ double s[2][W];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < count; i += kDiffReduceThreads) {
    const double2 p = partial[i];
    a += p.x;
    b += p.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  if (lane == 0) {
    s[0][warp] = a;
    s[1][warp] = b;
  }
  __syncthreads();
  if (warp < 2) {
    double v = s[warp][lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) {
      if (warp == 1 && count > 0) v *= sigma_in > 0.0 ? scale_in : diff_dscale(alpha, diff_sigma(sigma_in, sc));
      grad[warp] = v;
    }
  }
}

}  // namespace

int diff_grid(int n, int num_sms) { return std::max(1, std::min((n + kDiffThreads - 1) / kDiffThreads, num_sms * 8)); }

cudaError_t launch_diff_rows(int n, int bits, double sigma, const float* rgb, const GraphBufs& gb,
                             const DevScalars* sc, const DiffBufs& db, float4* x, int num_sms, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(k_diff_rows, dim3(diff_grid(n, num_sms)), dim3(kDiffThreads), 0, stream, false, n, bits, sigma,
                       diff_cexp(sigma), gb.pk, gb.c4, gb.perm1, rgb, sc, db, x);
}

cudaError_t launch_diff_rows_t(int n, int bits, double sigma, const float* grad, const GraphBufs& gb,
                               const DevScalars* sc, const DiffBufs& db, float4* u, int num_sms, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(k_diff_rows_t, dim3(diff_grid(n, num_sms)), dim3(kDiffThreads), 0, stream, false, n, bits,
                       sigma, diff_cexp(sigma), gb.c4, gb.perm1, grad, sc, db, u);
}

cudaError_t launch_diff_scatter(int n, const float4* x, const int32_t* perm1, float* out, int num_sms,
                                cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(k_diff_scatter, dim3(diff_grid(n, num_sms)), dim3(kDiffThreads), 0, stream, false, n, x, perm1,
                       out);
}

cudaError_t launch_diff_step(int n, float alpha, const GraphBufs& gb, const DiffBufs& db, const float4* src,
                             float4* dst, float* out, int num_sms, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(out ? k_diff_step<true> : k_diff_step<false>, dim3(diff_grid(n, num_sms)), dim3(kDiffThreads),
                       0, stream, false, n, alpha, gb.c4, db.r2, db.r4, src, dst, gb.perm1, out);
}

cudaError_t launch_diff_back_step(int n, float alpha, bool first, const GraphBufs& gb, const DiffBufs& db,
                                  const float4* x, const float4* u, float4* u_out, float* grad_in, double2* partial,
                                  int num_sms, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(grad_in ? k_diff_back_step<true> : k_diff_back_step<false>, dim3(diff_grid(n, num_sms)),
                       dim3(kDiffThreads), 0, stream, false, n, alpha, first, gb.c4, db, x, u, u_out, gb.perm1,
                       grad_in, partial);
}

cudaError_t launch_diff_reduce(int count, float alpha, double sigma, const DevScalars* sc, const double2* partial,
                               double* grad, cudaStream_t stream) {
  return launch_kernel(k_diff_reduce, dim3(1), dim3(kDiffReduceThreads), 0, stream, false, count, alpha, sigma,
                       diff_dscale(alpha, sigma), sc, partial, grad);
}

}  // namespace fgbd
