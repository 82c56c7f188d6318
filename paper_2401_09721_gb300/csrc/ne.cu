// NE-GBP: noise estimation using graph-based patches (Section 2.3), plus the
// per-point colour spread that the limited region of FSLR uses (Section 2.4).
//
// k_gather_colors: colours of the caller (input order) into sorted order.
// k_ne_moments: per point, its patch {i} + neighbours.  The spread
//   (sigma_R + sigma_G + sigma_B)/3 is written for every point.  A point with
//   exactly 6 neighbours contributes the patch a_i = [f_i, f_n1, ..., f_n6],
//   neighbours in increasing distance (ties by offset (dz, dy, dx), then
//   index), to the first and second moments sum a and sum a a^T.  uint8
//   colours are centred on 128 (exact in float16), so the moments are exact
//   integer sums: mma.sync products with float32 partial sums, moved to int64
//   before they can lose a bit (gram_mma.cuh).
// k_ne_finalize: one block.  Sigma = S2/N - mu mu^T in float64; float32
//   eigenvector estimates from a Householder tridiagonalisation, Sturm
//   multisection and inverse iteration (tridiag.cuh); each eigenvalue is then
//   the float64 Rayleigh quotient v^T Sigma v / v^T v, whose error is second
//   order in the eigenvector error; the values are sorted descending and the
//   tail rule gives sigma_est.
#include <algorithm>
#include <atomic>
#include <climits>

#include "eigen.cuh"
#include "gram_mma.cuh"
#include "select.cuh"
#include "tridiag.cuh"

namespace fgbd {
namespace {

constexpr int kTiles = 28;  // 3x3 output tiles covering the upper triangle of a 21x21 matrix

// Colours into sorted order, on their own (a whole run takes them in the link launch).
__global__ void __launch_bounds__(256) k_gather_colors(ColorArgs a, int n) {
  pdl_wait();
  for (int k0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x); k0 < n; k0 += 4 * gridDim.x * blockDim.x)
    colors_quad(a, k0, n);
}

__device__ __forceinline__ void tile_rc(int tile, int& r0, int& c0) {
  // tiles (ti, tj), ti <= tj, of a 7x7 grid of 3x3 blocks, row-major
  int ti = 0, rem = tile;
  while (rem >= 7 - ti) {
    rem -= 7 - ti;
    ++ti;
  }
  r0 = 3 * ti;
  c0 = 3 * (ti + rem);
}

// Float colours: the moments of a block or a group, the kTiles tiles (row-major),
// sum a, then the patch count; and where entry (r, c), r <= c, of sum a a^T is.
constexpr int kNeSums = 9 * kTiles + kD + 1;
__device__ __forceinline__ int tile_entry(int r, int c) {
  const int ti = r / 3, tj = c / 3;
  return 9 * (ti * 7 - ti * (ti - 1) / 2 + (tj - ti)) + 3 * (r % 3) + c % 3;
}

constexpr int kNeWarps = kNeThreads / 32;
// uint8 colours: one row of float16 a patch (gram_mma.cuh, patch-major): 28 columns
// of the seven nodes, four of zeros, and eight of padding (80-byte rows: the eight
// rows of an ldmatrix tile fall in distinct banks)
constexpr int kHRow = 40;
constexpr int kHPatches = 32;
constexpr int kRowFloats = 36;  // 32 float entries and padding: rows start on 16 bytes, four banks apart

// A patch place per neighbour, four bits each: its rank in the strict order (d^2,
// sorted id) from the 15 pairwise comparisons.  Starts from the link order, which
// the "w/o sort" ablation keeps: C1 prev, C1 next, C2 prev, C2 next, C3 prev, C3
// next.
__device__ __forceinline__ uint32_t patch_ranks(uint32_t wk, const uint32_t (&code)[6], const int (&nb)[6], int bits,
                                                bool sorted) {
  uint32_t ranks = 0x543210u;
  if (!sorted) return ranks;
  int kx, ky, kz;
  decode_c1(wk, bits, kx, ky, kz);
  unsigned long long key[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    int x, y, z;
    decode_c1(code[j], bits, x, y, z);
    const int dx = x - kx, dy = y - ky, dz = z - kz;
    key[j] = ((unsigned long long)uint32_t(dx * dx + dy * dy + dz * dz) << 32) | uint32_t(nb[j]);
  }
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i + 1; j < 6; ++j)
      if (key[j] < key[i]) ranks += (1u << (4 * i)) - (1u << (4 * j));
  return ranks;
}

// a node of a float16 patch: the colours of a packed word centred on 128 and `last`
// (0 or 1), from the bytes put into the fraction of 1024 (exact: 1024 + c - 1152)
__device__ __forceinline__ uint2 patch_node(uint32_t c, uint32_t last) {
  const __half2 off = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));  // 1152
  const uint32_t a = __byte_perm(c, 0x64646464u, 0x4140), b = __byte_perm(c, 0x64806464u + (last << 16), 0x7642);
  const __half2 ha = __hsub2(*reinterpret_cast<const __half2*>(&a), off);
  const __half2 hb = __hsub2(*reinterpret_cast<const __half2*>(&b), off);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&ha), *reinterpret_cast<const uint32_t*>(&hb));
}

// Per point: FSLR spread over the point and its neighbours (written to
// spread[k]) and, for a point with exactly 6 neighbours, its patch (the point
// then its neighbours by (d^2, dz, dy, dx, index)) written to the warp's patch
// block: row `lane` of float16 (uint8), column `lane` of float32 rows (float).
// Returns whether a patch was written.  Equal distances are ordered by sorted id
// alone: the C1 order is that of (z, y, x, input index).

// uint8 colours
__device__ __forceinline__ bool point_patch_u8(const MomentArgs& ma, int k, int lane, __half* ath) {
  const int n = ma.n, bits = ma.bits;
  const uint2 own = ma.pc[k];
  const int4 s = ma.c4[k];
  const uint32_t wk = own.x;  // packed code, with the same-line variant's missing-C1-link bits
  int nb[6];
  bool v[6];
  slots6(k, n, wk, s, nb, v);
  uint32_t code[6], c[6];
  int deg = 0;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const uint2 q = v[j] ? ma.pc[nb[j]] : make_uint2(0u, 0u);  // (an absent neighbour adds nothing below)
    code[j] = q.x;
    c[j] = q.y;
    deg += v[j];
  }
  ma.x0[k] = make_float4(float(own.y & 255u), float((own.y >> 8) & 255u), float((own.y >> 16) & 255u),
                         __uint_as_float(wk));
  // per channel the seven values in two words, their sum and sum of squares by
  // byte dot products
  const uint32_t t0 = __byte_perm(own.y, c[0], 0x5140), t1 = __byte_perm(c[1], c[2], 0x5140),
                 t2 = __byte_perm(c[3], c[4], 0x5140);  // (R, R, G, G) of two points
  const uint32_t u0 = __byte_perm(own.y, c[0], 0x7362), u1 = __byte_perm(c[1], c[2], 0x7362),
                 u2 = __byte_perm(c[3], c[4], 0x7362);  // (B, B, 0, 0)
  const uint32_t ra = __byte_perm(t0, t1, 0x5410), rb = __byte_perm(t2, c[5], 0x7410);
  const uint32_t ga = __byte_perm(t0, t1, 0x7632), gb = __byte_perm(t2, c[5], 0x7532);
  const uint32_t ba = __byte_perm(u0, u1, 0x5410), bb = __byte_perm(u2, c[5], 0x7610);
  const uint32_t ones = 0x01010101u;
  const int nn = deg + 1;
  // nn^2 times a population variance, an exact integer
  const auto var = [&](uint32_t a, uint32_t b) {
    const int sum = int(__dp4a(a, ones, __dp4a(b, ones, 0u))), sq = int(__dp4a(a, a, __dp4a(b, b, 0u)));
    return float(nn * sq - sum * sum);
  };
  // the mean of the three standard deviations is (sum of their roots) / (3 nn),
  // with one rounded reciprocal instead of four divisions (a few ulp in all, far
  // inside the band in which the selection decides exactly)
  ma.spread[k] = (sqrtf(var(ra, rb)) + sqrtf(var(ga, gb)) + sqrtf(var(ba, bb))) * __frcp_rn(3.0f * float(nn));
  if (deg != 6) return false;
  const uint32_t ranks = patch_ranks(wk, code, nb, bits, ma.sorted_patches != 0);
  uint2* row = reinterpret_cast<uint2*>(ath + lane * kHRow);
  row[0] = patch_node(own.y, 1u);
#pragma unroll
  for (int j = 0; j < 6; ++j) row[1 + ((ranks >> (4 * j)) & 15u)] = patch_node(c[j], 0u);
  return true;
}

// float colours
__device__ __forceinline__ bool point_patch_f32(const MomentArgs& ma, int k, int lane, float* atf) {
  const int n = ma.n, bits = ma.bits;
  const float4 own = ma.yf[k];
  const int4 s = ma.c4[k];
  const uint32_t wk = __float_as_uint(own.w);
  int nb[6];
  bool v[6];
  slots6(k, n, wk, s, nb, v);
  float4 q[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) q[j] = v[j] ? ma.yf[nb[j]] : own;
  int deg = 0;
#pragma unroll
  for (int j = 0; j < 6; ++j) deg += v[j];
  float mr = own.x, mg = own.y, mb = own.z;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    if (v[j]) {
      mr += q[j].x;
      mg += q[j].y;
      mb += q[j].z;
    }
  }
  const float icnt = __frcp_rn(float(deg + 1));
  mr *= icnt;
  mg *= icnt;
  mb *= icnt;
  float vr = (own.x - mr) * (own.x - mr), vg = (own.y - mg) * (own.y - mg), vb = (own.z - mb) * (own.z - mb);
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    if (v[j]) {
      vr += (q[j].x - mr) * (q[j].x - mr);
      vg += (q[j].y - mg) * (q[j].y - mg);
      vb += (q[j].z - mb) * (q[j].z - mb);
    }
  }
  ma.spread[k] = (sqrtf(vr * icnt) + sqrtf(vg * icnt) + sqrtf(vb * icnt)) * (1.0f / 3.0f);
  if (deg != 6) return false;
  uint32_t code[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) code[j] = __float_as_uint(q[j].w);
  const uint32_t ranks = patch_ranks(wk, code, nb, bits, ma.sorted_patches != 0);
  atf[0 * kRowFloats + lane] = own.x - 128.f;
  atf[1 * kRowFloats + lane] = own.y - 128.f;
  atf[2 * kRowFloats + lane] = own.z - 128.f;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    float* row = atf + (3u + 3u * ((ranks >> (4 * j)) & 15u)) * kRowFloats + lane;
    row[0] = q[j].x - 128.f;
    row[kRowFloats] = q[j].y - 128.f;
    row[2 * kRowFloats] = q[j].z - 128.f;
  }
  return true;
}

// the six Gram blocks into the block's int64 sums (sum a a^T, sum a, the patch count)
__device__ __forceinline__ void flush8(float (&gc)[6][4], int lane, unsigned long long* tot) {
#pragma unroll
  for (int t = 0; t < 6; ++t)
    gram_flush_nodes<kK + 1>(gc[t], t / 4, t < 4 ? t : t - 2, lane, tot, tot + kD * kD, tot + kD * kD + kD);
}

// Warp-synchronous: each warp takes 32 points at a time, stages their patches
// in its own shared-memory block and accumulates the moments with __syncwarp
// only.  The kernel is bound by its instructions (64 % of the issue slots used at 1M
// points), so neighbours are one 8-byte load of (code, colour), a patch is seven
// 8-byte stores, sums of squares are byte dot products and equal distances need
// no tie key: 36 -> 27 us at 1M points (x_0 as 16-byte neighbour loads: 31, and the
// link launch that writes it 9 us longer).  uint8 colours: float16 patches and
// mma.sync on the tensor pipe
// (gram_mma.cuh): per 16 patches six m16n8k16 products cover the upper triangle
// of the Gram matrix of (a, 1) in its 28 columns, moved to exact int64 sums every
// kGramFlushPatches patches.  Float colours: lanes 0..27 own one 3x3
// tile of the upper triangle of sum a a^T, four patches a load, and lanes 0..20
// one entry of sum a, in fp32 over 4 batches, then float64.  The block combines
// its warps through shared atomics and adds its totals to the context (uint8) or
// writes them (float); the last block of a group of kNeGroup to do so adds up the
// group's sums in block order, so that the eigen step reads a few rows instead of
// one a block (adding 608 rows there, one load after another, made the estimate
// launch 146 us at 217k points; with the groups it is 41 us).
template <int DT>
__device__ __forceinline__ void ne_moments_body(const MomentArgs& ma, int bid, int nblk) {
  const int n = ma.n;
  double* __restrict__ f64_partials = ma.f64_partials;
  DevScalars* __restrict__ sc = ma.sc;
  constexpr int kP = kD * kD + kD + 1;
  __shared__ __align__(16) __half s_h[DT == 0 ? kNeWarps : 1][kHPatches * kHRow];
  __shared__ __align__(16) float s_atf[DT == 1 ? kNeWarps : 1][kD * kRowFloats];
  __shared__ unsigned long long s_tot8[DT == 0 ? kP : 1];
  // (float: the warps' sums take the place of their patches when those are done)
  static_assert(sizeof(double) * kNeSums <= sizeof(float) * kD * kRowFloats, "a warp's sums fit its patch block");

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (DT == 0) {
    for (int i = threadIdx.x; i < kP; i += kNeThreads) s_tot8[i] = 0ull;
    // the columns behind the nodes stay zero
    *reinterpret_cast<uint2*>(&s_h[warp][lane * kHRow + 4 * (kK + 1)]) = make_uint2(0u, 0u);
  }
  // the graph's Eq. 4 exponent scale, once, for the filter steps that follow
  // (float64 work, here off their critical path)
  if (bid == 0 && threadIdx.x == 0 && !sc->cexp_ready) {
    sc->cexp = step_cexp(sc);
    __threadfence();
    sc->cexp_ready = 1u;
  }
  __syncthreads();
  int r0 = 0, c0 = 0;
  if (DT == 1 && lane < kTiles) tile_rc(lane, r0, c0);
  float gc[6][4] = {};  // uint8: the Gram blocks (m0, n0) .. (m0, n3), (m1, n2), (m1, n3)
  float accf[9] = {}, acc1f = 0.f;
  double accd[9] = {}, acc1d = 0.0;
  unsigned long long npatch = 0;
  int since_flush = 0;
  __half* ath = &s_h[DT == 0 ? warp : 0][0];
  float* atf = &s_atf[DT == 1 ? warp : 0][0];
  const uint32_t hbase = uint32_t(__cvta_generic_to_shared(ath));

  // uint8: each block takes a run of consecutive points, whose neighbours then lie in
  // this SM's L1 (step_run).  Float: the points are shared out over ma.shares shares,
  // four an SM, that take turns every 256 points, and a warp's float32 sums cover up
  // to four of its turns: what they round depends on the shares, so these stay as they
  // are while fewer blocks are resident (three an SM, without spills).  A block takes
  // its own share and, from the other end, one of those left over, where the turns are
  // fewest (217k points: 27 us, a launch of all the shares as blocks 34).
#pragma unroll 1
  for (int pass = 0; pass < (DT == 1 ? 2 : 1); ++pass) {
    const int share = pass == 0 ? bid : 2 * nblk - 1 - bid;
    if (DT == 1 && share >= ma.shares) break;
    const int2 run = DT == 0 ? step_run(n, bid, nblk, ma.per_sm) : make_int2(share * kNeThreads, n);
    const int stride = DT == 0 ? kNeThreads : ma.shares * kNeThreads;
    for (int base = run.x + warp * 32; base < run.y; base += stride) {
      const int k = base + lane;
      bool has = false;
      if (k < run.y) has = DT == 0 ? point_patch_u8(ma, k, lane, ath) : point_patch_f32(ma, k, lane, atf);
      if (!has) {
        if (DT == 0) {
          uint2* row = reinterpret_cast<uint2*>(ath + lane * kHRow);
#pragma unroll
          for (int j = 0; j < kK + 1; ++j) row[j] = make_uint2(0u, 0u);
        } else {
#pragma unroll
          for (int r = 0; r < kD; ++r) atf[r * kRowFloats + lane] = 0.f;
        }
      }
      if (DT == 1) npatch += __popc(__ballot_sync(0xffffffffu, has));
      __syncwarp();
      if (DT == 0) {
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          uint32_t lo[4], hi[4];
          ldsm_x4_trans(gram_patch_addr(hbase, 16 * ks, 0, kHRow, lane), lo);
          ldsm_x4_trans(gram_patch_addr(hbase, 16 * ks, 16, kHRow, lane), hi);
          mma_16816(gc[0], lo, lo[0], lo[2]);
          mma_16816(gc[1], lo, lo[1], lo[3]);
          mma_16816(gc[2], lo, hi[0], hi[2]);
          mma_16816(gc[3], lo, hi[1], hi[3]);
          mma_16816(gc[4], hi, hi[0], hi[2]);
          mma_16816(gc[5], hi, hi[1], hi[3]);
        }
        if (++since_flush == kGramFlushPatches / 32) {
          flush8(gc, lane, s_tot8);
          since_flush = 0;
        }
      } else {
        if (lane < kTiles) {
#pragma unroll 2
          for (int p = 0; p < 32; p += 4) {
            float4 a[3], b[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              a[i] = *reinterpret_cast<const float4*>(atf + (r0 + i) * kRowFloats + p);
              b[i] = *reinterpret_cast<const float4*>(atf + (c0 + i) * kRowFloats + p);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
              for (int j = 0; j < 3; ++j) {
                float t = accf[3 * i + j];
                t = fmaf(a[i].x, b[j].x, t);
                t = fmaf(a[i].y, b[j].y, t);
                t = fmaf(a[i].z, b[j].z, t);
                accf[3 * i + j] = fmaf(a[i].w, b[j].w, t);
              }
          }
        }
        if (lane < kD) {
          float sum = 0.f;
#pragma unroll
          for (int p = 0; p < 32; p += 4) {
            const float4 a = *reinterpret_cast<const float4*>(atf + lane * kRowFloats + p);
            sum += a.x;
            sum += a.y;
            sum += a.z;
            sum += a.w;
          }
          acc1f += sum;
        }
        if (++since_flush == 4) {
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            accd[i] += double(accf[i]);
            accf[i] = 0.f;
          }
          acc1d += double(acc1f);
          acc1f = 0.f;
          since_flush = 0;
        }
      }
      __syncwarp();
    }
    if (DT == 1) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        accd[i] += double(accf[i]);
        accf[i] = 0.f;
      }
      acc1d += double(acc1f);
      acc1f = 0.f;
      since_flush = 0;
    }
  }
  // combine the warps of the block
  if (DT == 0) {
    flush8(gc, lane, s_tot8);
    __syncthreads();
    for (int i = threadIdx.x; i < kP; i += kNeThreads) {
      const unsigned long long v = s_tot8[i];
      if (v == 0) continue;
      if (i < kD * kD) atomicAdd(reinterpret_cast<unsigned long long*>(&sc->s2[i]), v);
      else if (i < kD * kD + kD) atomicAdd(reinterpret_cast<unsigned long long*>(&sc->s1[i - kD * kD]), v);
      else atomicAdd(&sc->n_patches, v);
    }
    return;
  }
  double* own = reinterpret_cast<double*>(atf);
  if (lane < kTiles) {
#pragma unroll
    for (int i = 0; i < 9; ++i) own[9 * lane + i] = accd[i];
  }
  if (lane < kD) own[9 * kTiles + lane] = acc1d;
  if (lane == 0) own[9 * kTiles + kD] = double(npatch);
  __syncthreads();
  double* row = f64_partials + size_t(bid) * kNeSums;
  for (int i = threadIdx.x; i < kNeSums; i += kNeThreads) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kNeWarps; ++w) t += reinterpret_cast<const double*>(&s_atf[DT == 1 ? w : 0][0])[i];
    row[i] = t;
  }
  // the last block of the group adds up its rows, in block order, into the first
  const int g = bid / kNeGroup, b0 = g * kNeGroup, members = min(kNeGroup, nblk - b0);
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&sc->ne_groups[g], 1u) == uint32_t(members - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int i = threadIdx.x; i < kNeSums; i += kNeThreads) {
    double t = 0.0;
#pragma unroll 8
    for (int b = 0; b < members; ++b) t += __ldcg(&f64_partials[size_t(b0 + b) * kNeSums + i]);
    f64_partials[size_t(b0) * kNeSums + i] = t;
  }
}

template <int DT>
__global__ void __launch_bounds__(kNeThreads, DT == 0 ? 4 : 3) k_ne_moments(MomentArgs a) {
  pdl_wait();
  ne_moments_body<DT>(a, blockIdx.x, gridDim.x);
}

template <int DT>
__global__ void __launch_bounds__(kNeThreads, DT == 0 ? 4 : 3) k_ne_moments_seg(const __grid_constant__ Seg<MomentArgs> s) {
  pdl_wait();
  const int f = seg_frame(s, blockIdx.x);
  ne_moments_body<DT>(s.a[f], blockIdx.x - s.start[f], s.start[f + 1] - s.start[f]);
}

// ---------------------------------------------------------------- finalize

constexpr int kFinThreads = 384;      // 12 warps

// barriers of the first kFinThreads threads of a block (barrier 1; 0 is __syncthreads)
__device__ __forceinline__ void fin_bar() { asm volatile("bar.sync 1, %0;" ::"n"(kFinThreads) : "memory"); }

struct FinBar {
  __device__ void operator()() const { fin_bar(); }
};

// The eigenvalues of the D x D covariance S (float64, row-major in shared
// memory; Sf its float32 copy) as float64 Rayleigh quotients of float32
// eigenvector estimates (tridiag.cuh), sorted descending, then the tail rule:
// sigma_est and the eigenvalues into the context's scalars.  Threads
// 0..kFinThreads-1 of the block.
template <int D>
__device__ void eig_tail(const double* __restrict__ S, const float* __restrict__ Sf, DevScalars* __restrict__ sc,
                         double* __restrict__ sigma_out, int dtype) {
  static_assert(D <= 32, "warp 0 holds one eigenvalue a lane");
  __shared__ float V[D * D];  // eigenvector estimates (columns)
  __shared__ float s_mu[D];   // their float32 eigenvalues (the fallback of a non-finite quotient)
  __shared__ TridiagSmem<D, kFinThreads> tw;
  __shared__ long long s_key[D];
  __shared__ double s_sorted[D];
  constexpr int PR = (D + 1) / 2;  // pairs of rows (r, D - 1 - r)
  __shared__ double s_num[D][PR], s_den[D][PR];
  __shared__ double V64[D][D + 1];
  const int tid = threadIdx.x;

  // float32 eigenvector estimates: Householder tridiagonalisation, Sturm
  // multisection and inverse iteration (tridiag.cuh)
  eig_vectors_f32<D, kFinThreads>(Sf, tw, V, s_mu, FinBar{});
  if (tid == 0) atomicExch(&sc->sigma_near, 1u);  // (8 us to go)

  // float64 Rayleigh quotients of the eigenvector estimates.  This GPU has few
  // float64 lanes, so the numerators use the symmetry: v^T S v = sum_r v_r (S_rr
  // v_r + 2 sum_{c > r} S_rc v_c), a thread for rows r and D - 1 - r of one
  // vector, D - 1 off-diagonal terms whichever r (7500 -> 3700 cycles).
  for (int e = tid; e < D * D; e += kFinThreads) V64[e / D][e % D] = double(V[e]);
  fin_bar();
  static_assert(D * PR <= kFinThreads && (D & 1), "one pair a thread; the middle row pairs with itself");
  if (tid < D * PR) {
    const int k = tid / PR, r1 = tid % PR, r2 = D - 1 - r1;
    const int n1 = D - 1 - r1, total = r2 > r1 ? D - 1 : n1;
    double acc = 0.0, t1 = 0.0;
#pragma unroll 4
    for (int i = 0; i < D - 1; ++i) {
      if (i == n1) {
        t1 = acc;
        acc = 0.0;
      }
      const int r = i < n1 ? r1 : r2, c = i < n1 ? r1 + 1 + i : r2 + 1 + (i - n1);
      if (i < total) acc = fma(S[r * D + c], V64[c][k], acc);
    }
    const double t2 = n1 < D - 1 ? acc : 0.0, v1 = V64[r1][k], v2 = r2 > r1 ? V64[r2][k] : 0.0;
    if (n1 == D - 1) t1 = acc;
    s_num[k][r1] = v1 * fma(2.0, t1, S[r1 * D + r1] * v1) + v2 * fma(2.0, t2, S[r2 * D + r2] * v2);
    s_den[k][r1] = fma(v1, v1, v2 * v2);
  }
  fin_bar();
  // the rest runs in warp 0, lane j < D holding eigenvalue j
  if (tid < 32) {
    constexpr unsigned kFull = 0xffffffffu;
    const int lane = tid;
    double lam = 0.0;
    if (lane < D) {
      double n0 = 0.0, n1 = 0.0, d0 = 0.0, d1 = 0.0;
#pragma unroll
      for (int r = 0; r < PR; r += 2) {
        n0 += s_num[lane][r];
        d0 += s_den[lane][r];
        if (r + 1 < PR) {
          n1 += s_num[lane][r + 1];
          d1 += s_den[lane][r + 1];
        }
      }
      lam = div_newton(n0 + n1, d0 + d1);
      if (!isfinite(lam)) lam = double(s_mu[lane]);
    }
    // eigenvalues below 1e-9 max(lambda_1, 1) are numerical zeros (a rank-deficient
    // covariance); they are set to exactly 0 so the tail rule never decides on rounding noise
    double top = lane < D ? lam : -1.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(kFull, top, o));
    if (lane < D && fabs(lam) < kZeroEigRel * fmax(top, 1.0)) lam = 0.0;
    // descending order (ties by index), by counting the larger values
    // (float64 compares are slow here: the values are compared through
    // order-preserving 64-bit integer keys of their bit patterns)
    if (lane < D) s_key[lane] = order_key(lam);
    __syncwarp();
    if (lane < D) {
      const long long mine = order_key(lam);
      int rank = 0;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const long long o = s_key[j];
        rank += (o > mine) || (o == mine && j < lane);
      }
      s_sorted[rank] = lam;
    }
    __syncwarp();
    const double sorted = lane < D ? s_sorted[lane] : 0.0;
    if (lane < D) sc->eig[lane] = sorted;
    // tail sums lambda_j + ... + lambda_D by a suffix scan (a tail of exact
    // zeros sums to exactly 0 in any order)
    double suffix = sorted;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double t = __shfl_down_sync(kFull, suffix, o);
      if (lane + o < D) suffix += t;
    }
    // tail rule, every m tested at once: the smallest m with
    // mean(lambda_{m+1..D}) <= median(lambda_{m+1..D}), tested as
    // sum <= median * count; m = D - 1 always passes
    bool pass = false;
    if (lane < D) {
      const int cnt = D - lane;
      const double med = (cnt & 1) ? s_sorted[lane + cnt / 2]
                                   : 0.5 * (s_sorted[lane + cnt / 2 - 1] + s_sorted[lane + cnt / 2]);
      pass = suffix <= med * double(cnt);
    }
    const int m = __ffs(__ballot_sync(kFull, pass)) - 1;
    const double tail = __shfl_sync(kFull, suffix, m);
    if (lane == 0) {
      const double tau = div_newton(tail, double(D - m));
      const double sg = sqrt(fmax(tau, 0.0));
      sc->m = m;
      sc->tau = tau;
      sc->sigma_est = sg;
      sc->ne_valid = 1;
      // the selection's FSLR threshold of this sigma_est, formed here where it
      // is off the critical path (float64)
      fslr_band(sc->fslr_factor, sg, dtype, sc->fslr_thr);
      sc->fslr_ready = 1u;
      if (sigma_out) *sigma_out = sg;
      __threadfence();
      atomicExch(&sc->sigma_ready, 1u);
    }
  }
}

// sigma_est from the patch moments, by the first kFinThreads threads of one
// block (its barriers count those threads only, so the rest of a larger block
// may leave at once).  With sc->pooled_patch, the per-channel patches of
// D = 7 pooled over the channels (a reading of Section 2.3), built from the
// same sums: channel c's sums are the entries 3i + c of the RGB moments.
__device__ __noinline__ void finalize_block(int dtype, const double* __restrict__ f64_partials, int nblocks,
                                            DevScalars* __restrict__ sc, double* __restrict__ sigma_out) {
  __shared__ double S[kD * kD];
  __shared__ float Sf[kD * kD];  // Sigma rounded to float32 once, for the float32 work
  __shared__ double s_sum[kD * kD + kD + 1];
  __shared__ double s_tile[kNeSums];

  const int tid = threadIdx.x;
  constexpr int kT = kD / 3;  // points of a patch: the pooled dimension
  // gather the moments
  double npd;
  if (dtype == 0) {
    for (int i = tid; i < kD * kD; i += kFinThreads) s_sum[i] = double(sc->s2[i]);
    for (int i = tid; i < kD; i += kFinThreads) s_sum[kD * kD + i] = double(sc->s1[i]);
    if (tid == 0) s_sum[kD * kD + kD] = double(sc->n_patches);
  } else {
    for (int i = tid; i < kNeSums; i += kFinThreads) {
      double t = 0.0;  // the groups' sums, each in its first block's row
#pragma unroll 8
      for (int b = 0; b < nblocks; b += kNeGroup) t += f64_partials[size_t(b) * kNeSums + i];
      s_tile[i] = t;
    }
    fin_bar();
    for (int i = tid; i < kD * kD; i += kFinThreads) {
      const int r = i / kD, c = i % kD;
      s_sum[i] = r <= c ? s_tile[tile_entry(r, c)] : 0.0;
    }
    for (int i = tid; i <= kD; i += kFinThreads) s_sum[kD * kD + i] = s_tile[9 * kTiles + i];
  }
  fin_bar();
  npd = s_sum[kD * kD + kD];
  if (tid == 0 && dtype == 1) sc->n_patches = (unsigned long long)npd;
  if (npd < 1.0) {
    if (tid < kD) sc->eig[tid] = 0.0;
    if (tid == 0) {
      sc->tau = 0.0;
      sc->sigma_est = 0.0;
      sc->m = 0;
      sc->ne_valid = 1;
      if (sigma_out) *sigma_out = 0.0;
      __threadfence();
      atomicExch(&sc->sigma_near, 1u);
      atomicExch(&sc->sigma_ready, 1u);
    }
    return;
  }
  if (!sc->pooled_patch) {
    // Sigma = S2/N - mu mu^T: the upper triangle, one entry a thread, mirrored; 1/N
    // from one warp (a float64 division in every warp is 2500 cycles here)
    __shared__ double s_inv;
    if (tid == 0) s_inv = div_newton(1.0, npd);
    fin_bar();
    const double inv_n = s_inv;
    static_assert(kD * (kD + 1) / 2 <= kFinThreads, "one entry a thread");
    if (tid < kD * (kD + 1) / 2) {
      int r = 0, rest = tid;
      while (rest >= kD - r) {
        rest -= kD - r;
        ++r;
      }
      const int c = r + rest;
      const double v = fma(s_sum[r * kD + c], inv_n, -(s_sum[kD * kD + r] * inv_n) * (s_sum[kD * kD + c] * inv_n));
      S[r * kD + c] = S[c * kD + r] = v;
      Sf[r * kD + c] = Sf[c * kD + r] = float(v);
    }
    fin_bar();
    eig_tail<kD>(S, Sf, sc, sigma_out, dtype);
    return;
  }
  // pooled: 3 N samples of kT entries; mu_i = sum_c s1[3i + c] / 3N,
  // Sigma_ij = sum_c s2[3i + c][3j + c] / 3N - mu_i mu_j
  const double inv_3n = 1.0 / (3.0 * npd);
  for (int e = tid; e < kT * kT; e += kFinThreads) {
    const int i = e / kT, j = e % kT;
    const int lo = min(i, j), hi = max(i, j);
    double s2 = 0.0, mi = 0.0, mj = 0.0;
    for (int c = 0; c < 3; ++c) {
      s2 += s_sum[(3 * lo + c) * kD + 3 * hi + c];
      mi += s_sum[kD * kD + 3 * i + c];
      mj += s_sum[kD * kD + 3 * j + c];
    }
    const double v = s2 * inv_3n - (mi * inv_3n) * (mj * inv_3n);
    S[e] = v;
    Sf[e] = float(v);
  }
  fin_bar();
  eig_tail<kT>(S, Sf, sc, sigma_out, dtype);
}

__global__ void __launch_bounds__(kFinThreads) k_ne_finalize(int dtype, const double* __restrict__ f64_partials,
                                                           int nblocks, DevScalars* __restrict__ sc,
                                                           double* __restrict__ sigma_out) {
  pdl_wait();
  finalize_block(dtype, f64_partials, nblocks, sc, sigma_out);
}

// One block per SM (1024 threads of 64 registers fill its register file, so the
// rest of the SM's memory is L1 for the steps): block 0 computes sigma_est on an SM of its own, the others meanwhile take the first
// filter steps, which need the graph and the colours only.  With a.fuse they
// then also select and filter: they stop stepping once sigma_est is published
// (or after kSpecSure steps, then waiting for it) and run the selection over
// the stored steps (select_filter), so no second launch follows.
constexpr int kSpecThreads = 1024;

// FUSE: the selection and filter follow in the same launch (a.fuse); a kernel
// of its own, so that the plain launch carries none of their registers.
template <bool FUSE>
__global__ void __launch_bounds__(kSpecThreads, 1)
    k_ne_finalize_spec(int dtype, const double* __restrict__ f64_partials, int nblocks, DevScalars* __restrict__ sc,
                       double* __restrict__ sigma_out, FilterArgs a) {
  pdl_wait();
  __shared__ int s_ok;
  __shared__ int s_go;
  __shared__ float s_cexp;
  if (blockIdx.x == 0) {
    if (threadIdx.x < kFinThreads) finalize_block(dtype, f64_partials, nblocks, sc, sigma_out);
    return;
  }
  uint32_t epoch = 0;
  const int S = speculative_steps(a, a.spec_depth, 1, gridDim.x - 1, FUSE ? 1 : kSpecSure,
                                  FUSE ? &sc->sigma_ready : &sc->sigma_near, epoch, &s_ok, &s_cexp, &s_go);
  if (!FUSE || S < 0) return;
  // sigma_est of block 0 (a bounded wait)
  if (threadIdx.x == 0) {
    const unsigned long long t0 = global_ns();
    const unsigned long long limit = sc->wait_limit_ns;
    int ok = 1;
    while (!ld_acquire_u32(&sc->sigma_ready)) {
      if (global_ns() - t0 > limit) {
        atomicOr(&sc->status, kFlagTimeout);
        ok = 0;
        break;
      }
      __nanosleep(128);
    }
    s_ok = ok;
  }
  __syncthreads();
  if (!s_ok) return;
  select_filter<kSpecThreads>(a, S, 1, gridDim.x - 1, &sc->spec_barrier, epoch, 1);
}

// Segmented estimate launch (one block per SM, cooperative): block f < count
// computes sigma_est of frame f, and frame f's share of the other blocks takes
// its speculative filter steps (no fused selection here).
struct EstimateSeg {
  FilterArgs spec[kSegMax];
  const double* f64_partials[kSegMax];
  int nblocks[kSegMax];
  int first[kSegMax + 1];  // frame f's step blocks: [count + first[f], count + first[f + 1])
  int count;
};

__global__ void __launch_bounds__(kSpecThreads, 1) k_ne_finalize_spec_seg(const __grid_constant__ EstimateSeg e) {
  pdl_wait();
  __shared__ int s_ok;
  __shared__ int s_go;
  __shared__ float s_cexp;
  if (int(blockIdx.x) < e.count) {
    const int f = blockIdx.x;
    if (threadIdx.x < kFinThreads) finalize_block(e.spec[f].dtype, e.f64_partials[f], e.nblocks[f], e.spec[f].sc, nullptr);
    return;
  }
  const int b = int(blockIdx.x) - e.count;
  int f = 0;
  while (f + 1 < e.count && e.first[f + 1] <= b) ++f;
  uint32_t epoch = 0;
  speculative_steps(e.spec[f], e.spec[f].spec_depth, e.count + e.first[f], uint32_t(e.first[f + 1] - e.first[f]),
                    kSpecSure, nullptr, epoch, &s_ok, &s_cexp, &s_go);
}

// testing: the float64 quotient of the eigen step beside CUDA's own division
__global__ void __launch_bounds__(256) k_debug_div(const double* __restrict__ a, const double* __restrict__ b,
                                                   double* __restrict__ q_newton, double* __restrict__ q_div,
                                                   int64_t n) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    q_newton[i] = div_newton(a[i], b[i]);
    q_div[i] = a[i] / b[i];
  }
}

}  // namespace

cudaError_t launch_debug_div(const double* a, const double* b, double* q_newton, double* q_div, int64_t n,
                             cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int grid = int(std::min<int64_t>((n + 255) / 256, 152 * 8));
  return launch_kernel(k_debug_div, dim3(grid), dim3(256), 0, stream, false, a, b, q_newton, q_div, n);
}

cudaError_t launch_ne_moments_seg(const MomentArgs* a, int count, int dtype, int num_sms, cudaStream_t stream) {
  if (count < 1 || count > kSegMax) return cudaErrorInvalidValue;
  Seg<MomentArgs> sg;
  int blocks[kSegMax];
  // uint8 (exact sums, whatever blocks add them): the frames share the blocks that
  // fill the GPU once, so that a block's set-up and its 275 global atomics serve
  // several batches of points (16 frames of 20k-100k points: 65 -> 30 us).  Float: as many blocks as the one-frame launch has,
  // whose sums are the same bits.
  double total = 0.0;
  for (int f = 0; f < count; ++f) total += double(std::max(a[f].n, 0));
  const int fill = ne_moment_blocks(INT_MAX, num_sms, dtype);
  for (int f = 0; f < count; ++f) {
    sg.a[f] = a[f];
    sg.a[f].shares = ne_moment_shares(a[f].n, num_sms);
    blocks[f] = a[f].n > 0 ? ne_moment_blocks(a[f].n, num_sms, dtype) : 0;
    if (dtype == 0 && blocks[f] > 0)
      blocks[f] = std::max(1, std::min(blocks[f], int(double(fill) * double(a[f].n) / total)));
  }
  const int grid = seg_layout(sg, blocks, count);
  if (grid == 0) return cudaSuccess;
  if (dtype == 0) return launch_kernel(k_ne_moments_seg<0>, dim3(grid), dim3(kNeThreads), 0, stream, false, sg);
  return launch_kernel(k_ne_moments_seg<1>, dim3(grid), dim3(kNeThreads), 0, stream, false, sg);
}

cudaError_t launch_ne_finalize_seg(const FilterArgs* spec, const double* const* f64_partials, const int* nblocks,
                                   int count, int num_sms, cudaStream_t stream) {
  if (count < 1 || count > kSegMax || num_sms < 2 * count) return cudaErrorInvalidValue;
  EstimateSeg es;
  es.count = count;
  // the step blocks in proportion to the frames' points, at least one each
  const int pool = num_sms - count;
  double total = 0.0;
  for (int f = 0; f < count; ++f) total += double(std::max(spec[f].n, 1));
  int given = 0;
  es.first[0] = 0;
  for (int f = 0; f < count; ++f) {
    es.spec[f] = spec[f];
    es.f64_partials[f] = f64_partials[f];
    es.nblocks[f] = nblocks[f];
    const int left = count - 1 - f;  // frames after this one keep one block each
    int b = int(double(pool) * double(std::max(spec[f].n, 1)) / total);
    b = std::max(1, std::min(b, pool - given - left));
    if (f == count - 1) b = pool - given;
    given += b;
    es.first[f + 1] = given;
  }
  return launch_kernel(k_ne_finalize_spec_seg, dim3(count + pool), dim3(kSpecThreads), 0, stream, true, es);
}

cudaError_t launch_gather_colors(const ColorArgs& a, int n, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int grid = std::min((n + 1023) / 1024, 152 * 8);  // four points a thread
  return launch_kernel(k_gather_colors, dim3(grid), dim3(256), 0, stream, false, a, n);
}

// float colours: the shares of the points (k_ne_moments), at most two a block
int ne_moment_shares(int n, int num_sms) {
  const int need = int((int64_t(n) + kNeThreads - 1) / kNeThreads);
  return std::max(1, std::min({need, num_sms * 4, kNeGroup * kNeGroups}));
}

int ne_moment_blocks(int n, int num_sms, int dtype) {
  // resident blocks per SM, queried once (the same code runs on every device of one build)
  struct PerSm {
    int u8 = 1, f32 = 1;
  };
  static const PerSm per_sm = [] {
    PerSm p;
    int a = 0, b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_ne_moments<0>, kNeThreads, 0) == cudaSuccess && a > 0)
      p.u8 = a;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_ne_moments<1>, kNeThreads, 0) == cudaSuccess && b > 0)
      p.f32 = b;
    cudaGetLastError();
    return p;
  }();
  const int need = int((int64_t(n) + kNeThreads - 1) / kNeThreads);
  if (dtype == 0) return std::max(1, std::min(need, num_sms * per_sm.u8));
  const int shares = ne_moment_shares(n, num_sms);
  return std::max(1, std::min(shares, std::max(num_sms * per_sm.f32, (shares + 1) / 2)));
}

cudaError_t launch_ne_moments(const MomentArgs& a, int dtype, int num_sms, cudaStream_t stream) {
  if (a.n <= 0) return cudaSuccess;
  const int grid = ne_moment_blocks(a.n, num_sms, dtype);
  if (dtype == 0) {
    MomentArgs m = a;
    m.per_sm = grid % num_sms == 0 ? grid / num_sms : 1;
    return launch_kernel(k_ne_moments<0>, dim3(grid), dim3(kNeThreads), 0, stream, false, m);
  }
  MomentArgs m = a;
  m.shares = ne_moment_shares(a.n, num_sms);
  return launch_kernel(k_ne_moments<1>, dim3(grid), dim3(kNeThreads), 0, stream, false, m);
}

cudaError_t launch_ne_finalize(int dtype, const double* f64_partials, int nblocks, DevScalars* sc,
                               double* sigma_out, const FilterArgs* spec, int num_sms, cudaStream_t stream) {
  if (!spec || spec->spec_depth <= 0 || spec->n <= 0 || num_sms < 2)
    return launch_kernel(k_ne_finalize, dim3(1), dim3(kFinThreads), 0, stream, false, dtype, f64_partials, nblocks,
                         sc, sigma_out);
  if (spec->fuse)
    return launch_kernel(k_ne_finalize_spec<true>, dim3(num_sms), dim3(kSpecThreads), 0, stream, true,
                         dtype, f64_partials, nblocks, sc, sigma_out, *spec);
  return launch_kernel(k_ne_finalize_spec<false>, dim3(num_sms), dim3(kSpecThreads), 0, stream, true,
                       dtype, f64_partials, nblocks, sc, sigma_out, *spec);
}

}  // namespace fgbd
