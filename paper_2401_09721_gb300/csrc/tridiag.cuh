// Eigenvector estimates of the patch covariance for the noise estimate
// (Section 2.3), which needs the eigenvalues only.
//
// The eigenvalues themselves are the float64 Rayleigh quotients
// v^T Sigma v / v^T v of the vectors computed here (done by the caller): their
// error is second order in the vector error, so float32 vectors give
// eigenvalues far inside the noise estimate's tolerance.  The vectors come
// from the textbook route for a small dense symmetric matrix, in float32:
//   1. Householder reduction to tridiagonal form T = Q^T A Q (D - 2
//      reflections H_k = I - u_k u_k^T / h_k) in one warp, a column of A in a
//      lane's registers (two for D > 32);
//   2. the eigenvalues of T by Sturm-count multisection (every participating
//      thread counts the sign changes of the leading minors at its own point, so
//      each pass narrows every bracket at once; no iteration depends on
//      convergence);
//   3. one eigenvector of T per eigenvalue by two steps of inverse iteration
//      (an LDL^T solve of T - mu I), one thread each;
//   4. back to A's basis: v = H_0 H_1 ... H_{D-3} z.
// Within a cluster of eigenvalues closer than float32 resolution the vectors
// may mix, but each quotient then lies inside the cluster, so the eigenvalues
// stay within the cluster's width.  If a quotient is not finite the caller
// falls back to the multisection value, which is within float32 resolution.
#pragma once

#include "fgbd_internal.cuh"

namespace fgbd {
namespace {

// Shared-memory workspace of eig_vectors_f32<D, NT>.
template <int D, int NT>
struct TridiagSmem {
  static constexpr int kPer = NT / D;  // multisection points per eigenvalue and pass
  static constexpr int kPad = (D + 3) / 4 * 4;
  alignas(16) float U[D > 2 ? D - 2 : 1][kPad];  // reflection vectors u_k (rows)
  alignas(16) float sx[kPad], sp[kPad];          // the step's x and p: broadcast copies in the reduction
  float ih[D];                         // 1 / h_k, h_k = |u_k|^2 / 2 (0: no reflection)
  float d[D], e[D];                    // T: diagonal, off-diagonal e_i = T[i][i+1]
  float ds[D], e2s[D];                 // d_i and e_i^2 of T scaled by 2^-k to a size of one
  float2 br[D];                        // brackets (lo, hi] of the eigenvalues, ascending order
  float x[NT];                         // multisection points of one pass
  int cnt[NT];                         // their Sturm counts
  float P[D][D];                       // inverse iteration: reciprocal LDL^T pivots, [i][eigenvalue]
  float bounds[2];                     // Gershgorin interval of T
  float scale;                         // max |A_ii|: the size of the matrix
  float shrink;                        // the 2^-k above
};

// Number of eigenvalues of T below x, as the sign changes of the leading minors
// of T - x I, p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (Sturm's sequence): two
// dependent operations a row where the pivots' recurrence has a division (82
// cycles a row).  T and x come scaled to a size of one, and the pair of minors is
// scaled by a power of two every four rows, so that neither leaves float32's
// range.  A minor that is exactly zero counts one change with the two beside it,
// whatever its sign; the e_i^2 are at least 1e-16 (a change of T below the float32
// rounding of its size), so the pair stays above 1e-32 over four rows, never both zero.
template <int D>
__device__ __forceinline__ int sturm_count(const float* __restrict__ d, const float* __restrict__ e2, float x) {
  float p = d[0] - x, pp = 1.f;
  uint32_t c = __float_as_uint(p) >> 31;
#pragma unroll 1
  for (int i0 = 1; i0 < D; i0 += 4) {
#pragma unroll
    for (int i = i0; i < i0 + 4; ++i) {
      if (i < D) {
        const float q = fmaf(d[i] - x, p, -(e2[i - 1] * pp));
        c += (__float_as_uint(q) ^ __float_as_uint(p)) >> 31;
        pp = p;
        p = q;
      }
    }
    // the larger of the two to [1, 2)
    const int ex = int((__float_as_uint(fmaxf(fabsf(p), fabsf(pp))) >> 23) & 255u);
    const float f = __uint_as_float(uint32_t(min(max(254 - ex, 1), 254)) << 23);
    p *= f;
    pp *= f;
  }
  return int(c);
}

// passes of the bracket multisection until every bracket is below 2^-24 of
// the first interval: (NT + 1) (per + 1)^passes >= 2^24
__host__ __device__ constexpr int multisection_passes(int nt, int per) {
  double w = double(nt + 1);
  int p = 0;
  while (w < 16777216.0 && p < 24) {
    w *= double(per + 1);
    ++p;
  }
  return p;
}

// Eigenvector estimates of the symmetric D x D matrix As (shared memory,
// row-major float32), written to V (column k belongs to the k-th smallest
// eigenvalue of the reduced matrix; row-major, stride D); mu[k] receives that
// eigenvalue (float32 resolution).  Run by threads 0..NT-1 of the block;
// `bar` synchronises exactly those threads.  D <= NT.
//
// The loops over the reduction steps, the multisection passes, the inverse
// iterations and the reflections run as loops: unrolled, their straight-line
// code (tens of thousands of instructions, each executed once) is fetched
// faster than it issues only from the instruction cache, which it overflows.
// The loops over matrix entries inside them are unrolled, so the rows and
// vectors stay in registers.
template <int D, int NT, typename Bar>
__device__ void eig_vectors_f32(const float* __restrict__ As, TridiagSmem<D, NT>& w, float* __restrict__ V,
                                float* __restrict__ mu, Bar bar) {
  static_assert(D >= 1 && D <= NT && D <= 64, "one warp reduces the matrix; one thread per eigenvalue");
  constexpr int R = (D + 31) / 32;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  constexpr unsigned kFull = 0xffffffffu;

  // ---- 1. Householder reduction, in warp 0.  Lane j holds column j of A from
  // row k down (the registers move up one row a step).  Step k reads row k as
  // column k below the diagonal; x reaches every lane through shared memory,
  // every lane then forms |x|^2, and beside that chain its A x; u = x - alpha e_1
  // with alpha = -sign(x_0) |x| gives A u = A x - alpha A e_1.  A second exchange
  // hands p = A u / h to every lane, which forms u^T p itself: no warp reduction
  // and two exchanges a step (870 cycles at D = 21; rows spread over twelve warps with
  // warp reductions and block barriers took 1100).
  if (tid < 32) {
    float a[R][D];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int col = r * 32 + lane;
#pragma unroll
      for (int i = 0; i < D; ++i) a[r][i] = col < D ? As[i * D + col] : 0.f;
    }
    float scale = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int col = r * 32 + lane;
      if (col < D) scale = fmaxf(scale, fabsf(As[col * D + col]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) scale = fmaxf(scale, __shfl_xor_sync(kFull, scale, o));
    const float skip = 1e-12f * scale;  // a column below this size is taken as already reduced
    constexpr int N = D - 1;            // entries of x: rows k + 1 .., zero behind the last
    constexpr int Q = (N + 3) / 4;
    // (behind the last entry the copies hold zeros up to their padding)
    for (int i = lane; i < TridiagSmem<D, NT>::kPad; i += 32) w.sx[i] = w.sp[i] = 0.f;
    __syncwarp();
    // entry i of a vector over the columns below k, zero behind the last column
    const auto publish = [&](float* to, int k, const float (&val)[R]) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int col = r * 32 + lane;
        if (col < D) to[col > k ? col - k - 1 : D - 1 - k + col] = col > k ? val[r] : 0.f;  // (all of 0 .. D - 1)
      }
    };
#pragma unroll 1
    for (int k = 0; k + 2 < D; ++k) {
      float own[R];
#pragma unroll
      for (int r = 0; r < R; ++r) own[r] = a[r][0];
      publish(w.sx, k, own);
      __syncwarp();
      // (x is read again below: the columns leave no registers for it)
      const float4* sx = reinterpret_cast<const float4*>(w.sx);
      float s4[4] = {0.f, 0.f, 0.f, 0.f}, p[R], t4[R][4];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int l = 0; l < 4; ++l) t4[r][l] = 0.f;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const float4 c4 = sx[i];
        const float c[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          if (4 * i + l >= N) continue;
          s4[l] = fmaf(c[l], c[l], s4[l]);
#pragma unroll
          for (int r = 0; r < R; ++r) t4[r][l] = fmaf(a[r][4 * i + l + 1], c[l], t4[r][l]);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) p[r] = (t4[r][0] + t4[r][1]) + (t4[r][2] + t4[r][3]);
      const float xs = (s4[0] + s4[1]) + (s4[2] + s4[3]);
      const float x0 = w.sx[0];
      // (the approximate root: a reflection to a few float32 roundings either way; xs = 0: NaN, no reflection)
      const float nx = xs * rsqrtf(xs);
      const bool reflect = nx > skip && xs > 0.f;  // the same for every lane
      const float alpha = x0 > 0.f ? -nx : nx;
      const float ih = reflect ? __frcp_rn(fmaf(-x0, alpha, xs)) : 0.f;
      const float u0 = x0 - alpha;
      float u[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int col = r * 32 + lane;
        u[r] = !reflect || col <= k ? 0.f : (col == k + 1 ? u0 : own[r]);
        if (col < D) w.U[k][col] = u[r];
        if (col == k) {
          w.d[k] = own[r];
          w.e[k] = reflect ? alpha : x0;
          w.ih[k] = ih;
        }
        p[r] = fmaf(-alpha, a[r][1], p[r]) * ih;
      }
      if (reflect) {
        publish(w.sp, k, p);
        __syncwarp();
        // K = u^T p / (2 h), q = p - K u, A <- A - u q^T - q u^T
        float v4[4] = {0.f, 0.f, 0.f, 0.f};
        const float4* sp = reinterpret_cast<const float4*>(w.sp);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          const float4 t = sp[i], c = sx[i];
          v4[0] = fmaf(i == 0 ? u0 : c.x, t.x, v4[0]);
          v4[1] = fmaf(c.y, t.y, v4[1]);
          v4[2] = fmaf(c.z, t.z, v4[2]);
          v4[3] = fmaf(c.w, t.w, v4[3]);
        }
        const float K = 0.5f * ((v4[0] + v4[1]) + (v4[2] + v4[3])) * ih;
        float qc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) qc[r] = fmaf(-K, u[r], p[r]);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          const float4 pv = sp[i], xv = sx[i];
          const float t[4] = {pv.x, pv.y, pv.z, pv.w}, c[4] = {i == 0 ? u0 : xv.x, xv.y, xv.z, xv.w};
#pragma unroll
          for (int l = 0; l < 4; ++l) {
            if (4 * i + l >= N) continue;
            const float q = fmaf(-K, c[l], t[l]);
#pragma unroll
            for (int r = 0; r < R; ++r)
              a[r][4 * i + l] = fmaf(-c[l], qc[r], fmaf(-q, u[r], a[r][4 * i + l + 1]));
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) a[r][D - 1] = 0.f;
        __syncwarp();  // x and p have been read
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
          for (int i = 0; i < N; ++i) a[r][i] = a[r][i + 1];
          a[r][D - 1] = 0.f;
        }
        __syncwarp();  // x has been read
      }
    }
    // the last two rows
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int col = r * 32 + lane;
      if (col == D - 2) w.d[D - 2] = a[r][0];
      if (col == D - 1) {
        w.e[D - 2] = a[r][0];
        w.d[D - 1] = a[r][1];
        w.e[D - 1] = 0.f;
      }
    }
    if (lane == 0) w.scale = scale;
    __syncwarp();
    // Gershgorin interval of T
    float glo = 3.0e38f, ghi = -3.0e38f;
    for (int i = lane; i < D; i += 32) {
      const float rad = fabsf(w.e[i]) + (i > 0 ? fabsf(w.e[i - 1]) : 0.f);
      glo = fminf(glo, w.d[i] - rad);
      ghi = fmaxf(ghi, w.d[i] + rad);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      glo = fminf(glo, __shfl_xor_sync(kFull, glo, o));
      ghi = fmaxf(ghi, __shfl_xor_sync(kFull, ghi, o));
    }
    const float pad = 1e-6f * fmaxf(fabsf(glo), fabsf(ghi)) + 1e-30f;
    // 2^-k of the interval's larger end: T and the points scaled by it have a size of one
    const int ex = int((__float_as_uint(fmaxf(fabsf(glo - pad), fabsf(ghi + pad))) >> 23) & 255u);
    const float shrink = __uint_as_float(uint32_t(min(max(254 - ex, 1), 254)) << 23);
    if (lane == 0) {
      w.bounds[0] = glo - pad;
      w.bounds[1] = ghi + pad;
      w.shrink = shrink;
    }
    for (int i = lane; i < D; i += 32) {
      const float es = w.e[i] * shrink;
      w.ds[i] = w.d[i] * shrink;
      w.e2s[i] = fmaxf(es * es, 1e-16f);
    }
    for (int i = lane; i < D; i += 32) w.br[i] = make_float2(glo - pad, ghi + pad);
  }
  bar();

  const float scale = w.scale;
  if (!(scale > 0.f)) {
    // the zero matrix: every eigenvalue is 0, any basis will do
    for (int i = tid; i < D * D; i += NT) V[i] = (i / D == i % D) ? 1.f : 0.f;
    for (int i = tid; i < D; i += NT) mu[i] = 0.f;
    bar();
    return;
  }
  const float shrink = w.shrink;

  // ---- 2. multisection.  Pass 0 counts at NT points across the whole
  // interval; a crossing between points t - 1 and t brackets the eigenvalues
  // k with cnt[t-1] <= k < cnt[t].  Later passes put kPer points in each
  // bracket.  (The counts do not decrease along x; if rounding ever made
  // them, an eigenvalue left without a new bracket keeps its old one.)
  {
    const float lo = w.bounds[0], hi = w.bounds[1];
    const float x = lo + (hi - lo) * (float(tid + 1) / float(NT + 1));
    w.x[tid] = x;
    w.cnt[tid] = sturm_count<D>(w.ds, w.e2s, x * shrink);
  }
  bar();
  {
    const int c = w.cnt[tid];
    const int c0 = tid == 0 ? 0 : w.cnt[tid - 1];
    const float x0 = tid == 0 ? w.bounds[0] : w.x[tid - 1];
    for (int k = max(c0, 0); k < min(c, D); ++k) w.br[k] = make_float2(x0, w.x[tid]);
    if (tid == NT - 1)
      for (int k = max(c, 0); k < D; ++k) w.br[k] = make_float2(w.x[tid], w.bounds[1]);
  }
  bar();
  constexpr int kPer = TridiagSmem<D, NT>::kPer;
  constexpr int kPasses = multisection_passes(NT, kPer);
  const bool sect = tid < D * kPer;
  const int sk = tid / kPer, sj = tid % kPer;
#pragma unroll 1
  for (int pass = 0; pass < kPasses; ++pass) {
    float2 b = make_float2(0.f, 0.f);
    if (sect) {
      b = w.br[sk];
      const float x = b.x + (b.y - b.x) * (float(sj + 1) / float(kPer + 1));
      w.x[tid] = x;
      w.cnt[tid] = sturm_count<D>(w.ds, w.e2s, x * shrink);
    }
    bar();
    if (sect) {
      // the first of the bracket's points whose count exceeds k sets the new
      // bracket; if none does, the last point and the old upper end
      const bool f = w.cnt[tid] > sk;
      const bool fp = sj > 0 && w.cnt[tid - 1] > sk;
      if (f && !fp) w.br[sk] = make_float2(sj == 0 ? b.x : w.x[tid - 1], w.x[tid]);
      else if (!f && sj == kPer - 1) w.br[sk] = make_float2(w.x[tid], b.y);
    }
    bar();
  }

  // ---- 3. inverse iteration, thread k for eigenvalue k; 4. back to A's basis
  if (tid < D) {
    const int k = tid;
    const float m = 0.5f * (w.br[k].x + w.br[k].y);
    mu[k] = m;
    const float tiny = scale * 5.9604645e-8f;  // 2^-24 of the matrix
    // LDL^T of T - m I, pivots guarded against tiny ones; P holds their
    // reciprocals (the same factors serve both iterations)
    {
      float piv = w.d[0] - m;
      if (fabsf(piv) < tiny) piv = piv < 0.f ? -tiny : tiny;
      float rp = __frcp_rn(piv);
      w.P[0][k] = rp;
#pragma unroll 4
      for (int i = 1; i < D; ++i) {
        piv = fmaf(-(w.e[i - 1] * rp), w.e[i - 1], w.d[i] - m);
        if (fabsf(piv) < tiny) piv = piv < 0.f ? -tiny : tiny;
        rp = __frcp_rn(piv);
        w.P[i][k] = rp;
      }
    }
    float z[D];
    // a start vector with no special direction: entries in [0.5, 1.5)
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const float f = float(i) * 0.61803398875f + float(k) * 0.41421356237f;
      z[i] = 0.5f + (f - floorf(f));
    }
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {
      // solve L D L^T y = z: forward with L (multipliers e_{i-1} / piv_{i-1}),
      // scale by D^-1, back with L^T
#pragma unroll
      for (int i = 1; i < D; ++i) z[i] = fmaf(-(w.e[i - 1] * w.P[i - 1][k]), z[i - 1], z[i]);
      z[D - 1] *= w.P[D - 1][k];
      float ymax = fabsf(z[D - 1]);
#pragma unroll
      for (int i = D - 2; i >= 0; --i) {
        const float rpi = w.P[i][k];
        z[i] = fmaf(-(w.e[i] * rpi), z[i + 1], z[i] * rpi);
        ymax = fmaxf(ymax, fabsf(z[i]));
      }
      // normalise (by the largest entry first, so the sum of squares cannot overflow)
      const float is = ymax > 0.f ? __frcp_rn(ymax) : 1.f;
      float ss = 0.f;
#pragma unroll
      for (int i = 0; i < D; ++i) {
        z[i] *= is;
        ss = fmaf(z[i], z[i], ss);
      }
      const float nrm = rsqrtf(ss);
#pragma unroll
      for (int i = 0; i < D; ++i) z[i] *= nrm;
    }
    // v = H_0 H_1 ... H_{D-3} z; u_s is zero in entries 0..s, so the
    // products run over all D entries
#pragma unroll 1
    for (int s = D - 3; s >= 0; --s) {
      const float ih = w.ih[s];
      if (!(ih > 0.f)) continue;
      float us[(D + 3) / 4 * 4];
#pragma unroll
      for (int i = 0; i < (D + 3) / 4; ++i) {
        const float4 t = reinterpret_cast<const float4*>(w.U[s])[i];
        us[4 * i] = t.x;
        us[4 * i + 1] = t.y;
        us[4 * i + 2] = t.z;
        us[4 * i + 3] = t.w;
      }
      float t0 = 0.f, t1 = 0.f, t2 = 0.f;
#pragma unroll
      for (int i = 0; i < D; i += 3) {
        t0 = fmaf(us[i], z[i], t0);
        if (i + 1 < D) t1 = fmaf(us[i + 1], z[i + 1], t1);
        if (i + 2 < D) t2 = fmaf(us[i + 2], z[i + 2], t2);
      }
      const float c = (t0 + t1 + t2) * ih;
#pragma unroll
      for (int i = 0; i < D; ++i) z[i] = fmaf(-c, us[i], z[i]);
    }
#pragma unroll
    for (int i = 0; i < D; ++i) V[i * D + k] = z[i];
  }
  bar();
}

}  // namespace
}  // namespace fgbd
