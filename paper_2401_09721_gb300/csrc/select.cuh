// FSLR selection (Eq. 6, Section 2.4) and the graph low-pass filter (Eq. 5)
// as one device routine, run by the blocks of a cooperative grid: the
// selection kernel (k_filter) and, inside the noise-estimate launch, the
// blocks that took the first steps while sigma_est was computed.
//
//   phase 0   the FSLR keep flag of each point (spread <= 2 sigma_est) goes to
//             keep8; the kept power sum y^2 and the kept count are reduced, and
//             so are the stored steps' per-point power sums x_q^2;
//             x_0 = y is written unless it is there or steps are stored.
//   J(1..S)   from those sums, by warp 0 of every block (the same values
//             everywhere: the sums are exact integers).
//   step t    x_t = x_{t-1}/2 + (sum_j e_j x_{t-1}[j]) / (2 sum_j e_j) with
//             e_j = exp(-(d2_j - min_j d2_j) / sigma_g^2) (eq5_step): the rows
//             of D^{-1} W of Eq. 4, normalised once per graph by step 1 (from
//             the neighbours' coordinates, carried in x.w) and read back by the
//             later steps.
//             In select mode the kept power sum x_t^2 is reduced and, after a
//             grid barrier, J(t) = |sigma^2 - (sum y^2 - sum x_t^2)/(3 N_sel)|;
//             the search stops at the first t with J(t) >= J(t-1), keeping
//             q* = t-1.
//   output    the kept iterate is gathered back to input order (optional).
// Data written earlier in the same launch by other blocks is read after a grid
// barrier that orders it (filter_step.cuh): the iterates through L1, what a step
// reads once (stored steps' sums, keep flags, sigma_est) from L2.
// Sums of squares are fixed-point integers (2^-8), so the reduction is exact
// and independent of the order in which blocks add.  Grid barriers have a 2 s
// wait limit; a block that gives up latches kFlagTimeout and every block
// returns.
#pragma once

#include <climits>

#include "filter_step.cuh"

namespace fgbd {
namespace {

// ---- float-float arithmetic (an unevaluated sum hi + lo of two floats,
// about 44 significant bits): the error-free transformations TwoSum (Knuth)
// and TwoProduct through a fused multiply-add, as in Dekker's double-length
// arithmetic.  Float64 is slow on this GPU; this stands in for it in the rare
// FSLR decisions that float32 cannot take.
struct FF {
  float hi, lo;
};
__device__ __forceinline__ FF ff_fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF ff_add(FF x, FF y) {
  const float s = __fadd_rn(x.hi, y.hi);
  const float bb = __fsub_rn(s, x.hi);
  const float e = __fadd_rn(__fsub_rn(x.hi, __fsub_rn(s, bb)), __fsub_rn(y.hi, bb));
  return ff_fast_two_sum(s, __fadd_rn(e, __fadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ FF ff_neg(FF x) { return {-x.hi, -x.lo}; }
__device__ __forceinline__ FF ff_mul(FF x, FF y) {
  const float p = __fmul_rn(x.hi, y.hi);
  const float e = fmaf(x.hi, y.hi, -p);
  return ff_fast_two_sum(p, fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, e)));
}
__device__ __forceinline__ FF ff_div_int(FF x, int k) {
  const float kf = float(k);
  const float q1 = __fdiv_rn(x.hi, kf);
  const FF r = ff_add(x, ff_neg(ff_mul({q1, 0.f}, {kf, 0.f})));
  return ff_fast_two_sum(q1, __fdiv_rn(r.hi, kf));
}
__device__ __forceinline__ FF ff_sqrt(FF x) {
  if (!(x.hi > 0.f)) return {0.f, 0.f};
  const float s = __fsqrt_rn(x.hi);
  const FF r = ff_add(x, ff_neg(ff_mul({s, 0.f}, {s, 0.f})));
  return ff_fast_two_sum(s, __fdiv_rn(r.hi, __fmul_rn(2.f, s)));
}

// The FSLR keep decision of Section 2.4, spread <= threshold, for a point whose
// float32 spread is too close to the threshold to decide.  The spread is the
// mean of the three population standard deviations over the point and its
// neighbours; the decision compares their sum with 3 thr (thr as float-float).
// uint8 colours: cnt^2 times each variance is the integer cnt sum x^2 - (sum x)^2
// (below 2^22, exact in float32), so only the three square roots need float-float.
// float colours: two-pass (mean, then squared deviations) in float-float.
__device__ __noinline__ bool keep_ff(const FilterArgs& a, int k, FF thr) {
  int nb[7];
  bool v[7];
  const uint32_t pkk = a.pk[k];
  nb[0] = k;
  v[0] = true;
  nb[1] = k - 1;
  v[1] = c1_prev_linked(pkk, k);
  nb[2] = k + 1;
  v[2] = c1_next_linked(pkk, k, a.n);
  const int4 s = a.c4[k];
  nb[3] = s.x;
  nb[4] = s.y;
  nb[5] = s.z;
  nb[6] = s.w;
#pragma unroll
  for (int j = 3; j < 7; ++j) v[j] = in_range(nb[j], a.n);
  int cnt = 0;
#pragma unroll
  for (int j = 0; j < 7; ++j) cnt += v[j];
  FF total = {0.f, 0.f};
  if (a.dtype == 0) {
    uint32_t c[7];
#pragma unroll
    for (int j = 0; j < 7; ++j) c[j] = v[j] ? a.y8[nb[j]] : 0u;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      int sx = 0, sq = 0;
#pragma unroll
      for (int j = 0; j < 7; ++j) {
        const int x = int((c[j] >> (8 * ch)) & 255u);
        sx += x;
        sq += x * x;
      }
      const int V = cnt * sq - sx * sx;  // cnt^2 var; absent neighbours read as 0 and add nothing
      total = ff_add(total, ff_sqrt({float(V), 0.f}));
    }
    // sum_c sqrt(V_c) / cnt against 3 thr
    const FF d = ff_add(total, ff_neg(ff_mul(thr, {3.f * float(cnt), 0.f})));
    return d.hi < 0.f || (d.hi == 0.f && d.lo <= 0.f);
  }
  float col[3][7];
#pragma unroll
  for (int j = 0; j < 7; ++j) {
    if (v[j]) {
      const float4 y = a.yf[nb[j]];
      col[0][j] = y.x;
      col[1][j] = y.y;
      col[2][j] = y.z;
    } else {
      col[0][j] = col[1][j] = col[2][j] = 0.f;
    }
  }
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) {
    FF sum = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 7; ++j)
      if (v[j]) sum = ff_add(sum, {col[ch][j], 0.f});
    const FF mean = ff_div_int(sum, cnt);
    FF ss = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 7; ++j) {
      if (v[j]) {
        const FF d = ff_add({col[ch][j], 0.f}, ff_neg(mean));
        ss = ff_add(ss, ff_mul(d, d));
      }
    }
    total = ff_add(total, ff_sqrt(ff_div_int(ss, cnt)));
  }
  const FF d = ff_add(total, ff_neg(ff_mul(thr, {3.f, 0.f})));
  return d.hi < 0.f || (d.hi == 0.f && d.lo <= 0.f);
}

// The same decision at a window w > 1: the point and its 6 + NX neighbour
// slots, in loops (only the few points in the float32 band come here).
template <int NX>
__device__ __noinline__ bool keep_ff_wide(const FilterArgs& a, int k, FF thr) {
  const int n = a.n;
  const uint32_t pkk = a.pk[k];
  const int4 s = a.c4[k];
  FF total = {0.f, 0.f};
  int cnt = 1;
#pragma unroll 1
  for (int j = 0; j < 6 + NX; ++j) cnt += neighbour_of(j, k, n, pkk, s, a.cx, a.cx_stride) >= 0;
  if (a.dtype == 0) {
    int sx[3], sq[3];
    const uint32_t own = a.y8[k];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      const int x = int((own >> (8 * ch)) & 255u);
      sx[ch] = x;
      sq[ch] = x * x;
    }
#pragma unroll 1
    for (int j = 0; j < 6 + NX; ++j) {
      const int o = neighbour_of(j, k, n, pkk, s, a.cx, a.cx_stride);
      if (o < 0) continue;
      const uint32_t c = a.y8[o];
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        const int x = int((c >> (8 * ch)) & 255u);
        sx[ch] += x;
        sq[ch] += x * x;
      }
    }
    // cnt^2 var <= 19^2 127.5^2 < 2^24: exact in float32
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) total = ff_add(total, ff_sqrt({float(cnt * sq[ch] - sx[ch] * sx[ch]), 0.f}));
    const FF d = ff_add(total, ff_neg(ff_mul(thr, {3.f * float(cnt), 0.f})));
    return d.hi < 0.f || (d.hi == 0.f && d.lo <= 0.f);
  }
#pragma unroll 1
  for (int ch = 0; ch < 3; ++ch) {
    const float* own = reinterpret_cast<const float*>(&a.yf[k]);
    FF sum = {own[ch], 0.f};
#pragma unroll 1
    for (int j = 0; j < 6 + NX; ++j) {
      const int o = neighbour_of(j, k, n, pkk, s, a.cx, a.cx_stride);
      if (o >= 0) sum = ff_add(sum, {reinterpret_cast<const float*>(&a.yf[o])[ch], 0.f});
    }
    const FF mean = ff_div_int(sum, cnt);
    FF dd = ff_add({own[ch], 0.f}, ff_neg(mean));
    FF ss = ff_mul(dd, dd);
#pragma unroll 1
    for (int j = 0; j < 6 + NX; ++j) {
      const int o = neighbour_of(j, k, n, pkk, s, a.cx, a.cx_stride);
      if (o < 0) continue;
      dd = ff_add({reinterpret_cast<const float*>(&a.yf[o])[ch], 0.f}, ff_neg(mean));
      ss = ff_add(ss, ff_mul(dd, dd));
    }
    total = ff_add(total, ff_sqrt(ff_div_int(ss, cnt)));
  }
  const FF d = ff_add(total, ff_neg(ff_mul(thr, {3.f, 0.f})));
  return d.hi < 0.f || (d.hi == 0.f && d.lo <= 0.f);
}

template <int NX>
__device__ __forceinline__ bool keep_ff_nx(const FilterArgs& a, int k, FF thr) {
  if constexpr (NX == 0) return keep_ff(a, k, thr);
  else return keep_ff_wide<NX>(a, k, thr);
}

__device__ __forceinline__ void write_out(const FilterArgs& a, int i, float4 x) {
  if (a.out_dtype == 0) {
    uint8_t* o = static_cast<uint8_t*>(a.out) + 3 * size_t(i);
    o[0] = uint8_t(fminf(fmaxf(rintf(x.x), 0.f), 255.f));
    o[1] = uint8_t(fminf(fmaxf(rintf(x.y), 0.f), 255.f));
    o[2] = uint8_t(fminf(fmaxf(rintf(x.z), 0.f), 255.f));
  } else {
    float* o = static_cast<float*>(a.out) + 3 * size_t(i);
    o[0] = x.x;
    o[1] = x.y;
    o[2] = x.z;
  }
}

// x_q of sorted point k, wherever the kept iterate is (kept_buf)
__device__ __forceinline__ float4 kept_value(const FilterArgs& a, int kept, int k) {
  if (kept < 0) return x0_of(a, k);
  if (kept == kKeptBest) return __ldcg(&a.xbest[k]);
  if (kept >= 2) return __ldcg(&a.spec_x[size_t(kept - 2) * size_t(a.cap) + k]);
  return __ldcg(&(kept ? a.xbuf1 : a.xbuf0)[k]);
}

// x_0 of the sorted points k0 .. k0 + 3 (k0 a multiple of 4; those at or past
// n only when `full` is false, and then left unread).  The packed coordinates
// (x.w) are read only when `with_pk`.
__device__ __forceinline__ void x0_quad(const FilterArgs& a, int k0, bool full, bool with_pk, float4 (&x)[4]) {
  uint32_t p[4] = {0u, 0u, 0u, 0u};
  if (with_pk) {
    if (full) {
      const uint4 v = *reinterpret_cast<const uint4*>(a.pk + k0);
      p[0] = v.x;
      p[1] = v.y;
      p[2] = v.z;
      p[3] = v.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (k0 + i < a.n) p[i] = a.pk[k0 + i];
    }
  }
  if (a.dtype == 0) {
    uint32_t y[4] = {0u, 0u, 0u, 0u};
    if (full) {
      const uint4 v = *reinterpret_cast<const uint4*>(a.y8 + k0);
      y[0] = v.x;
      y[1] = v.y;
      y[2] = v.z;
      y[3] = v.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (k0 + i < a.n) y[i] = a.y8[k0 + i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      x[i] = make_float4(float(y[i] & 255u), float((y[i] >> 8) & 255u), float((y[i] >> 16) & 255u),
                         __uint_as_float(p[i]));
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 c = (full || k0 + i < a.n) ? a.yf[k0 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
      x[i] = make_float4(c.x, c.y, c.z, __uint_as_float(p[i]));
    }
  }
}

// colours of the kept iterate at sorted point k (x.w is not meaningful)
__device__ __forceinline__ float4 kept_rgb(const FilterArgs& a, int kept, int k) {
  if (kept < 0) {
    float r, g, b;
    load_y(a, k, r, g, b);
    return make_float4(r, g, b, 0.f);
  }
  return kept_value(a, kept, k);
}

// The kept iterate in input order: input points i0 .. i0 + 3 per thread and
// trip, their sorted positions read as two int4 and the four gathers issued
// together; uint8 / float32 output as 32- / 128-bit stores where aligned.
__device__ __forceinline__ void output_quads(const FilterArgs& a, int kept, int gtid, int gstride) {
  const int n = a.n;
  const bool u8 = a.out_dtype == 0;
  const bool wide = (reinterpret_cast<uintptr_t>(a.out) & (u8 ? 3u : 15u)) == 0;
  for (int i0 = 4 * gtid; i0 < n; i0 += 4 * gstride) {
    const bool full = i0 + 4 <= n;
    int kk[4] = {-1, -1, -1, -1};
    if (full) {
      const int4 u = *reinterpret_cast<const int4*>(a.rank12 + i0);
      const int4 v = *reinterpret_cast<const int4*>(a.rank12 + i0 + 2);
      kk[0] = u.x;
      kk[1] = u.z;
      kk[2] = v.x;
      kk[3] = v.z;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i0 + i < n) kk[i] = a.rank12[i0 + i].x;
    }
    float4 v[4];
    bool ok[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      ok[i] = in_range(kk[i], n);
      v[i] = ok[i] ? kept_rgb(a, kept, kk[i]) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (full && wide && ok[0] && ok[1] && ok[2] && ok[3]) {
      if (u8) {
        uint32_t b[12];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          b[3 * i + 0] = uint32_t(fminf(fmaxf(rintf(v[i].x), 0.f), 255.f));
          b[3 * i + 1] = uint32_t(fminf(fmaxf(rintf(v[i].y), 0.f), 255.f));
          b[3 * i + 2] = uint32_t(fminf(fmaxf(rintf(v[i].z), 0.f), 255.f));
        }
        uint32_t* o = reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(a.out) + 3 * size_t(i0));
#pragma unroll
        for (int w = 0; w < 3; ++w)
          o[w] = b[4 * w] | (b[4 * w + 1] << 8) | (b[4 * w + 2] << 16) | (b[4 * w + 3] << 24);
      } else {
        float4* o = reinterpret_cast<float4*>(static_cast<float*>(a.out) + 3 * size_t(i0));
        o[0] = make_float4(v[0].x, v[0].y, v[0].z, v[1].x);
        o[1] = make_float4(v[1].y, v[1].z, v[2].x, v[2].y);
        o[2] = make_float4(v[2].z, v[3].x, v[3].y, v[3].z);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (ok[i] && i0 + i < n) write_out(a, i0 + i, v[i]);
    }
  }
}

// The selection and filter for the blocks [first, first + members) of a
// cooperative grid of THREADS-thread blocks, from S stored steps (0: none),
// grid barriers on *bar (epoch: the barriers this grid has passed on it), per_sm
// blocks on an SM;
// NX further neighbour slots per point (window w > 1: NX = 6 (w - 1)).
// DEEP: up to kSpecMax stored steps (else kSpecSure).  PART: the whole search, or (a
// segmented launch) leave it after step a.step_cap if it has not ended, or take it up there.
enum class SearchPart { kWhole, kCapped, kRest };
template <int THREADS, int NX = 0, bool DEEP = false, SearchPart PART = SearchPart::kWhole>
__device__ __forceinline__ void select_filter(const FilterArgs& a, int S, int first, uint32_t members,
                                              uint32_t* bar, uint32_t& epoch, int per_sm) {
  constexpr int W = THREADS / 32;
  static_assert(kSpecMax <= W && 3 + 2 * kSpecMax <= THREADS, "a warp or more a stored step, a thread a sum");
  constexpr int kSums = DEEP ? 5 : 3 + 2 * kSpecSure;
  __shared__ unsigned long long s_red[kSums * W];
  __shared__ int s_ok;
  const int n = a.n;
  const int gtid = (int(blockIdx.x) - first) * THREADS + int(threadIdx.x);
  const int gstride = int(members) * THREADS;
  DevScalars* sc = a.sc;
  constexpr bool kRest = PART == SearchPart::kRest;
  const bool select = kRest || a.mode == 0;
  // Block-uniform scalars, computed by thread 0: the FSLR threshold 2 sigma_est
  // as a float32 band [t_lo, t_hi] (outside it float32 decides) and as float-float.
  __shared__ float s_thr[4];
  if (threadIdx.x == 0 && select && !kRest) {
    if (a.sigma_src == &sc->sigma_est && sc->fslr_ready) {
      // as the eigen step formed them with sigma_est (fslr_band, the same arithmetic)
#pragma unroll
      for (int i = 0; i < 4; ++i) s_thr[i] = sc->fslr_thr[i];
    } else {
      fslr_band(a.fslr_factor, __ldcg(a.sigma_src), a.dtype, s_thr);
    }
  }
  __syncthreads();
  float t_lo = 0.f, t_hi = 0.f;
  FF thr = {0.f, 0.f};
  if (select && !kRest) {
    t_lo = s_thr[0];
    t_hi = s_thr[1];
    thr = {s_thr[2], s_thr[3]};
  }

  // ---- phase 0: keep flags and the Eq. 6 sums; x_0 = y unless the steps are stored.
  // Four consecutive points per thread and trip, read with 16-byte loads that
  // are all issued before the first is used.
  // The stored steps' power sums follow from the same flags.  Up to kSpecSure steps:
  // a thread takes its own quads again and holds the sums of every step.  DEEP: a
  // few warps a step, from the flags in shared memory, and two sums a thread, so
  // that eight steps cost as little as three (a 20,000-point frame with six or
  // seven steps: 13 us, where taking four of them after a grid barrier each took
  // 26).  On large frames, with two trips a block and three steps, the barriers
  // between flags and sums cost 2 us (1M points: 23.2 -> 25.7), so they keep the first.
  // acc: kept y^2, all y^2, kept count; then kept and all x_q^2 (DEEP: of this warp's step)
  unsigned long long acc[kSums] = {};
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool write_x0 = !S && !a.x0;
  const bool phase0 = !kRest && (select || write_x0);
  // (DEEP: blocks take equal runs of quads; with quads by thread number, three of
  // four blocks of a frame below a wave would have none)
  constexpr int kKeepTrips = DEEP ? 4 : 1;  // quads of keep flags a thread leaves between two barriers
  __shared__ uint32_t s_keep[DEEP ? kKeepTrips * THREADS : 1];
  const int quads = (n + 3) / 4, share = (quads + int(members) - 1) / int(members);
  const int qa = DEEP ? min(quads, (int(blockIdx.x) - first) * share) : gtid - int(threadIdx.x);
  const int qb = DEEP ? min(quads, qa + share) : quads;
  const int tile = DEEP ? kKeepTrips * THREADS : int(members) * THREADS;
  for (int qt = qa; phase0 && qt < qb; qt += tile) {
    const int qe = DEEP ? min(qb, qt + tile) : min(qb, qt + THREADS);
    for (int quad = qt + int(threadIdx.x); quad < qe; quad += THREADS) {
      const int k0 = 4 * quad;
      uint32_t kw = 0;
      const bool full = k0 + 4 <= n;
      float4 x[4];
      x0_quad(a, k0, full, write_x0, x);
      float sp[4] = {0.f, 0.f, 0.f, 0.f};
      if (select) {
        if (full) {
          const float4 v = *reinterpret_cast<const float4*>(a.spread + k0);
          sp[0] = v.x;
          sp[1] = v.y;
          sp[2] = v.z;
          sp[3] = v.w;
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (k0 + i < n) sp[i] = a.spread[k0 + i];
        }
      }
      if (write_x0) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (full || k0 + i < n) a.xbuf0[k0 + i] = x[i];
      }
      if (select) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (!full && k0 + i >= n) continue;
          bool keep;
          if (a.all_points || sp[i] <= t_lo) keep = true;
          else if (sp[i] > t_hi) keep = false;
          else keep = keep_ff_nx<NX>(a, k0 + i, thr);
          kw |= uint32_t(keep) << (8 * i);
          const unsigned long long q2 = sq3(x[i]);
          acc[1] += q2;
          if (keep) {
            acc[0] += q2;
            acc[2] += 1;
          }
        }
        if (full) {
          *reinterpret_cast<uint32_t*>(a.keep8 + k0) = kw;
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (k0 + i < n) a.keep8[k0 + i] = uint8_t((kw >> (8 * i)) & 1u);
        }
      }
      if constexpr (DEEP) s_keep[quad - qt] = kw;
    }
    if (DEEP && S > 0) {
      const int wq = W / S;  // warps a stored step
      __syncthreads();
      if (warp < wq * S) {
        const int32_t* zr = a.spec_z + size_t(warp % S) * size_t(a.cap);
#pragma unroll 4
        for (int quad = qt + 32 * (warp / S) + lane; quad < qe; quad += 32 * wq) {
          const int kz = 4 * quad;
          int4 z = make_int4(0, 0, 0, 0);
          if (kz + 4 <= n) {
            z = __ldcg(reinterpret_cast<const int4*>(zr + kz));
          } else {
            z.x = __ldcg(zr + kz);
            if (kz + 1 < n) z.y = __ldcg(zr + kz + 1);
            if (kz + 2 < n) z.z = __ldcg(zr + kz + 2);
          }
          const uint32_t f = s_keep[quad - qt];
          acc[4] += (unsigned long long)((long long)z.x + z.y + z.z + z.w);
          acc[3] += (unsigned long long)((long long)(f & 1u ? z.x : 0) + (f & 0x100u ? z.y : 0) +
                                         (f & 0x10000u ? z.z : 0) + (f & 0x1000000u ? z.w : 0));
        }
      }
      __syncthreads();
    }
  }
  if constexpr (!DEEP) {
    for (int k0 = 4 * gtid; !kRest && S > 0 && k0 < n; k0 += 4 * gstride) {
      const bool full = k0 + 4 <= n;
      uint32_t kw = 0;
      int32_t z[kSpecSure][4] = {};
      if (full) kw = *reinterpret_cast<const uint32_t*>(a.keep8 + k0);
#pragma unroll
      for (int q = 0; q < kSpecSure; ++q) {
        if (q < S) {
          const int32_t* zr = a.spec_z + size_t(q) * size_t(a.cap) + k0;
          if (full) {
            const int4 v = __ldcg(reinterpret_cast<const int4*>(zr));
            z[q][0] = v.x;
            z[q][1] = v.y;
            z[q][2] = v.z;
            z[q][3] = v.w;
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (k0 + i < n) z[q][i] = __ldcg(zr + i);
          }
        }
      }
      if (!full) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (k0 + i < n) kw |= uint32_t(a.keep8[k0 + i] != 0) << (8 * i);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool keep = (kw >> (8 * i)) & 1u;
#pragma unroll
        for (int q = 0; q < kSpecSure; ++q) {
          if (q < S) {
            const unsigned long long zz = (unsigned long long)(long long)z[q][i];
            acc[4 + 2 * q] += zz;
            if (keep) acc[3 + 2 * q] += zz;
          }
        }
      }
    }
  }
  if (select && !kRest) {
#pragma unroll
    for (int i = 0; i < kSums; ++i) {
      acc[i] = warp_sum(acc[i]);
      if (lane == 0) s_red[i * W + warp] = acc[i];
    }
    __syncthreads();
    const int t = threadIdx.x;
    if (t < 3 + 2 * S) {
      // sum t: over the warps, or (DEEP, a stored step's) over those that took it
      unsigned long long v = 0;
      if (!DEEP || t < 3) {
        for (int w = 0; w < W; ++w) v += s_red[t * W + w];
      } else {
        for (int w = (t - 3) >> 1; w < W / S * S; w += S) v += s_red[(4 - (t & 1)) * W + w];
      }
      unsigned long long* to = t == 0 ? &sc->ysq_keep : t == 1 ? &sc->ysq_all : &sc->n_keep;
      if (t >= 3)
        to = reinterpret_cast<unsigned long long*>(t & 1 ? &sc->spec_keep[(t - 1) / 2] : &sc->spec_all[(t - 2) / 2]);
      if (v) atomicAdd(to, v);
    }
  }
  if (phase0 && !grid_barrier(bar, &sc->status, members, epoch, &s_ok, sc)) return;

  // J(0..S) from the stored terms, by warp 0 of each block, a lane a step (every block
  // reaches the same values: the sums are exact integers).  Under the global
  // reading (a.q_global) the search never stops early and q* is the argmin of
  // J over 0..q_max (the smaller q among equal values); a new best iterate
  // beyond the stored steps is copied to xbest while the next step reads it.
  __shared__ int s_ctl[6];  // keep_all, q_limit, q_final, stop, q_best, copy the last iterate
  __shared__ float s_cexp;
  const bool global = select && a.q_global;
  // J(t) = |sigma^2 - lost_t / (3 N_sel)| with lost_t the exact fixed-point sum of
  // y^2 - x_t^2: sigma^2 and 2^-kSqShift / (3 N_sel) are formed once, so each J
  // is one fused multiply-add (float64 operations have a long latency here).  What
  // the later steps' J needs stays in shared memory, not in every thread's registers.
  __shared__ double s_sig2, s_inv3n, s_J_prev, s_J_best;
  __shared__ unsigned long long s_ysq;
  if (warp == 0) {
    // lane t: J(t) of the stored step t, all side by side; the scalars loaded
    // together (one round trip to L2)
    static_assert(kSpecMax < 32, "a lane a stored step");
    const uint32_t c_ready = sc->cexp_ready;
    const float c_val = sc->cexp;
    const int q_fixed = a.q_src ? min(max(*a.q_src, 0), kQCap) : a.q_fixed;
    const int q_limit = n == 0 ? 0 : (select ? a.q_max : q_fixed);
    int keep_all = 0, q_final = 0, stopped = 0, q_best = 0;
    if (select) {
      const double sigma = __ldcg(a.sigma_src);
      const unsigned long long nkt = ld_relaxed_u64(&sc->n_keep);
      const unsigned long long ysk = ld_relaxed_u64(&sc->ysq_keep);
      const unsigned long long ysa = ld_relaxed_u64(&sc->ysq_all);
      unsigned long long xk = 0, xa = 0;
      if (lane >= 1 && lane <= S) {
        xk = ld_relaxed_u64(reinterpret_cast<const unsigned long long*>(&sc->spec_keep[lane]));
        xa = ld_relaxed_u64(reinterpret_cast<const unsigned long long*>(&sc->spec_all[lane]));
      }
      keep_all = nkt == 0;  // no point left: every point is used
      const double nsel = keep_all ? double(n) : double(nkt);
      const unsigned long long ysq = keep_all ? ysa : ysk;
      const double sig2 = sigma * sigma;
      const double inv3n = (1.0 / double(1 << kSqShift)) / (3.0 * nsel);
      // sum of y^2 - x_t^2 over the points of Eq. 6: exact in two's complement
      const double lost = double((long long)(ysq - (keep_all ? xa : xk)));
      const int m = min(S, q_limit);
      double J = fabs(fma(-lost, inv3n, sig2));
      if (lane == 0) J = sig2;  // J(0): nothing filtered yet
      const double before = __shfl_up_sync(0xffffffffu, J, 1);
      const uint32_t up = __ballot_sync(0xffffffffu, !global && lane >= 1 && lane <= m && J >= before);
      stopped = up != 0;
      const int last = stopped ? __ffs(int(up)) - 1 : m;  // the last J of the search so far
      q_final = stopped ? last - 1 : m;
      double J_prev = __shfl_sync(0xffffffffu, J, q_final);
      if (kRest) {
        stopped = 0;
        q_final = sc->resume_t;
        J_prev = sc->J[q_final];
      }
      double J_best = sig2;
      if (global) {
        for (int t = 1; t <= m; ++t) {
          const double Jt = __shfl_sync(0xffffffffu, J, t);
          if (Jt < J_best) {
            J_best = Jt;
            q_best = t;
          }
        }
      }
      if (lane == 0) {
        s_sig2 = sig2;
        s_inv3n = inv3n;
        s_J_prev = J_prev;
        s_J_best = J_best;
        s_ysq = ysq;
      }
      if (!kRest && int(blockIdx.x) == first) {
        if (lane <= last) sc->J[lane] = J;
        if (lane == 0 && last > 0) sc->n_J = last + 1;
      }
    }
    if (lane == 0) {
      s_cexp = c_ready ? c_val : step_cexp(sc);
      s_ctl[0] = keep_all;
      s_ctl[1] = q_limit;
      s_ctl[2] = q_final;
      s_ctl[3] = stopped;
      s_ctl[4] = q_best;
      s_ctl[5] = 0;
    }
  }
  __syncthreads();
  const float cexp = s_cexp;
  const bool keep_all = s_ctl[0] != 0;
  const int q_limit = s_ctl[1];
  int q_final = s_ctl[2];
  const bool stopped = s_ctl[3] != 0;
  const int2 run = step_run(n, int(blockIdx.x) - first, int(members), per_sm);
  bool copy_best = false;  // this step's source is the best iterate so far: copy it to xbest
  for (int t = (kRest ? q_final : S) + 1; t <= q_limit && !stopped; ++t) {
    const float4* src =
        t == 1 && a.x0 ? a.x0
                       : (!kRest && S > 0 && t == S + 1) ? a.spec_x + size_t(S - 1) * size_t(a.cap)
                                                         : ((t & 1) ? a.xbuf0 : a.xbuf1);
    float4* dst = (t & 1) ? a.xbuf1 : a.xbuf0;
    unsigned long long loc = 0;
    for (int k = run.x + int(threadIdx.x); k < run.y; k += THREADS) {
      const StepHead h = step_head(a, src, k);
      const float4 xo =
          t == 1 ? eq5_step_nx<NX, true>(a, src, k, n, cexp, h) : eq5_step_nx<NX, false>(a, src, k, n, cexp, h);
      dst[k] = xo;
      if (copy_best) a.xbest[k] = h.xk;
      if (select && (keep_all || __ldcg(a.keep8 + k))) loc += sq3(xo);
    }
    if (select) {
      loc = block_sum_u64<THREADS>(loc, s_red);
      if (threadIdx.x == 0 && loc) atomicAdd(&sc->sumsq[t], loc);
    }
    // (the barrier starts with __syncthreads: every thread has read s_ctl[3])
    if (!grid_barrier(bar, &sc->status, members, epoch, &s_ok, sc)) return;
    if (select) {
      if (threadIdx.x == 0) {
        const unsigned long long ss = ld_relaxed_u64(&sc->sumsq[t]);
        const double lost = double((long long)(s_ysq - ss));
        const double J = fabs(fma(-lost, s_inv3n, s_sig2));
        if (gtid == 0) {
          sc->J[t] = J;
          sc->n_J = t + 1;
        }
        if (global) {
          const bool better = J < s_J_best;
          if (better) {
            s_J_best = J;
            s_ctl[4] = t;
          }
          s_ctl[3] = 0;
          s_ctl[5] = better;
        } else {
          s_ctl[3] = J >= s_J_prev;
          if (!(J >= s_J_prev)) s_J_prev = J;
        }
      }
      __syncthreads();
      if (s_ctl[3]) {
        q_final = t - 1;
        break;
      }
      q_final = t;
      copy_best = s_ctl[5] != 0;
      if (PART == SearchPart::kCapped && t == a.step_cap && t < q_limit) {
        if (gtid == 0) sc->resume_t = t;
        return;
      }
    } else {
      q_final = t;
    }
  }
  // where the kept iterate is (power 0: the colours themselves, since x_0 is in no
  // iterate buffer where the steps read it elsewhere)
  int kept = q_final == 0 ? -1 : q_final <= S ? 2 + q_final - 1 : (q_final & 1);
  if (global) {
    const int qb = s_ctl[4];
    if (qb == 0) kept = -1;
    else if (qb <= S) kept = 2 + qb - 1;
    else if (qb == q_final) kept = qb & 1;  // the last step: still in its buffer
    else kept = kKeptBest;                  // copied while step qb + 1 read it
    q_final = qb;
  }
  if (gtid == 0) {
    if (!a.q_src) sc->q_sel = q_final;
    sc->kept_buf = kept;
    if (select) sc->sel_valid = 1;
    if (select && q_limit == 0) sc->n_J = 1;
  }
  if (a.out) output_quads(a, kept, gtid, gstride);
}

}  // namespace
}  // namespace fgbd
