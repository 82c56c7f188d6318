// SLG: scan-line graph construction (Section 2.2).
//
// Sorting by a code of Eq. 1-3 is sorting by three b-bit coordinates, most
// significant first, with equal codes (repeated voxels) in input order.  The
// three orders are made side by side, each in two steps:
//   k_coord_hist      the three coordinate histograms: the size of every row,
//                     a row being the points of one most significant
//                     coordinate of a code (z for C1, x for C2, y for C3);
//   k_bucket_scatter  every point into its row of each code, in any order
//                     inside the row: a block ranks its tile's points with
//                     shared-memory counters and reserves its share of every
//                     row with one global atomic a row;
//   k_bucket_sort     the points of a window of consecutive rows (or of the
//                     lines of one large row that start in the window) ordered
//                     by (code, input index) in shared memory.
// C1 ends with the packed code of every sorted (C1) point, its input index and
// the rank of every input point; C2 and C3 with the input indices and the codes
// along the code, C2 also with the rank of every input point.
// k_link: points consecutive along a code are linked.  In C1 order the code-1
// neighbours are implicit (k-1, k+1); C2/C3 neighbours are written as slots;
// a pair already linked by an earlier code is left out so the union is a set,
// and each distinct edge's length is summed for sigma_g.
#include <algorithm>
#include <cstdlib>

#include "fgbd_internal.cuh"

namespace fgbd {
namespace {

// the coordinate rows of the histograms (0 x, 1 y, 2 z) that are the most and
// the second most significant of code c (0 C1, 1 C2, 2 C3); the least is row c
__device__ __forceinline__ int row_coord(int c) { return c == 0 ? 2 : c - 1; }
__device__ __forceinline__ int mid_coord(int c) { return c == 2 ? 0 : c + 1; }

// code c of a packed C1 code
__device__ __forceinline__ uint32_t code_from_c1(int c, uint32_t c1, int b, uint32_t m) {
  return c == 0 ? c1 : code_of(c, c1 & m, (c1 >> b) & m, c1 >> (2 * b), b);
}

// this warp's offset from the totals of the warps of the block (at most 32)
__device__ __forceinline__ uint32_t warps_before(const uint32_t* s_w, int lane, int warp) {
  return __reduce_add_sync(0xffffffffu, lane < warp ? s_w[lane] : 0u);
}

__device__ __forceinline__ uint32_t warp_inclusive(uint32_t x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// exclusive scan of one value per thread over the block (s_w: one word a warp)
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t* s_w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t x = warp_inclusive(v, lane);
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  return warps_before(s_w, lane, warp) + x - v;
}

// The three coordinate histograms, 1024-thread blocks (up to two per SM) taking
// whole 4096-point tiles of the input, merged with global atomics.
__device__ __forceinline__ void coord_hist_body(const HistArgs& a, int bid, int nblk) {
  __shared__ uint32_t h[3][kMaxRadix];
  const int radix = 1 << a.bits;
  const int tiles = (a.n + kSortTile - 1) / kSortTile;
  for (int i = threadIdx.x; i < 3 * kMaxRadix; i += blockDim.x) (&h[0][0])[i] = 0;
  const uint32_t m = uint32_t(radix) - 1u;
  // four consecutive points a thread (a tile is kSortTile = 4 x 1024 points),
  // read as three 16-byte loads where the array is aligned, all issued before
  // the first shared-memory atomic
  static_assert(kSortTile == 4 * 1024, "1024 threads take four points each");
  const bool vec = (reinterpret_cast<uintptr_t>(a.xyz) & 15u) == 0;
  bool bad = false;
  __syncthreads();
  for (int t = bid; t < tiles; t += nblk) {
    const int p0 = t * kSortTile + 4 * int(threadIdx.x);
    int c[12];
    if (vec && p0 + 4 <= a.n) {
      const int4* q = reinterpret_cast<const int4*>(a.xyz + 3 * size_t(p0));
      const int4 v0 = q[0], v1 = q[1], v2 = q[2];
      c[0] = v0.x; c[1] = v0.y; c[2] = v0.z; c[3] = v0.w;
      c[4] = v1.x; c[5] = v1.y; c[6] = v1.z; c[7] = v1.w;
      c[8] = v2.x; c[9] = v2.y; c[10] = v2.z; c[11] = v2.w;
    } else {
#pragma unroll
      for (int j = 0; j < 12; ++j) c[j] = p0 + j / 3 < a.n ? a.xyz[3 * size_t(p0) + j] : 0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (p0 + i >= a.n) break;
      const uint32_t xi = uint32_t(c[3 * i]), yi = uint32_t(c[3 * i + 1]), zi = uint32_t(c[3 * i + 2]);
      bad |= (xi > m) | (yi > m) | (zi > m);
      atomicAdd(&h[0][xi & m], 1u);
      atomicAdd(&h[1][yi & m], 1u);
      atomicAdd(&h[2][zi & m], 1u);
    }
  }
  if (bad) atomicOr(&a.sc->status, kFlagRange);
  __syncthreads();
  for (int c = 0; c < 3; ++c)
    for (int d = threadIdx.x; d < radix; d += blockDim.x)
      if (h[c][d]) atomicAdd(&a.sc->chist[c][d], h[c][d]);
}

__global__ void __launch_bounds__(1024, 2) k_coord_hist(HistArgs a) {
  pdl_wait();
  coord_hist_body(a, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(1024, 2) k_coord_hist_seg(const __grid_constant__ Seg<HistArgs> s) {
  pdl_wait();
  const int f = seg_frame(s, blockIdx.x);
  coord_hist_body(s.a[f], blockIdx.x - s.start[f], s.start[f + 1] - s.start[f]);
}

// ---------------------------------------------------------------- rows
// One tile of up to kSortTile points a block: (input index, code) of every
// point into its row of the three codes.  The order inside a row is left to
// k_bucket_sort, so the ranks come from shared-memory atomics instead of
// ballots, the tiles need no counts from an earlier launch (a block reserves
// its share of a row with one global atomic), and the three codes share one
// read of the coordinates.  A tile is staged in row order in shared memory
// before it is written, so that the points of one row leave as one run.
// Measured (1M body points, b = 10): 16 us for the three codes; one of the
// three ballot-ranked passes it stands in for took 17.5 us, and with its scan
// and counts 25.  It waits on its loads, barriers and shared-memory ranks (27 %
// of the issue slots used); scattering without staging (8-byte random writes)
// took 36 us.  Two blocks an SM: more and smaller tiles pay for the row scans
// and the global atomics (37 us with 608 blocks).
template <int THREADS>
struct ScatterShape {
  static constexpr int kKpt = kSortTile / THREADS;    // points per thread
  static constexpr int kDpt = kMaxRadix / THREADS;    // rows per thread
  static constexpr int kMinBlocks = 2;                // resident blocks per SM
  static_assert(kSortTile % THREADS == 0 && kMaxRadix % THREADS == 0, "points and rows divide evenly");
};
constexpr int kScatterThreads = 1024;  // the one-frame path (the batch tuner may pick 256 or 512)
// row counts (then write-out offsets), the tile's row starts, and the staged tile
constexpr size_t kScatterSmem = sizeof(uint32_t) * (6 * size_t(kMaxRadix)) + sizeof(uint2) * size_t(kSortTile);

template <int THREADS>
__device__ __forceinline__ void bucket_scatter_body(const BucketArgs& a, int t) {
  using SS = ScatterShape<THREADS>;
  constexpr int kKpt = SS::kKpt, kDpt = SS::kDpt, kWarps = THREADS / 32;
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t* s_cnt = smem;                                               // [3 coordinates][rows]
  uint32_t* s_at = s_cnt + 3 * kMaxRadix;                               // [3 coordinates][rows]
  uint2* s_pt = reinterpret_cast<uint2*>(s_at + 3 * kMaxRadix);         // [kSortTile]
  __shared__ uint32_t s_w[6][kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = a.bits, radix = 1 << b, n = a.n;
  const uint32_t m = uint32_t(radix) - 1u;
  const int base = t * a.tile, end = min(n, base + a.tile);

  uint32_t code[kKpt];
#pragma unroll
  for (int j = 0; j < kKpt; ++j) {
    const int i = base + j * THREADS + tid;
    code[j] = 0u;
    if (i < end) {
      const uint32_t x = uint32_t(a.xyz[3 * size_t(i)]) & m;
      const uint32_t y = uint32_t(a.xyz[3 * size_t(i) + 1]) & m;
      const uint32_t z = uint32_t(a.xyz[3 * size_t(i) + 2]) & m;
      code[j] = code_of(0, x, y, z, b);
    }
  }
  // the rows' sizes; this thread owns the consecutive rows tid * kDpt ..
  uint32_t size[3][kDpt], sum[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    sum[c] = 0u;
#pragma unroll
    for (int i = 0; i < kDpt; ++i) {
      const int d = tid * kDpt + i;
      size[c][i] = d < radix ? a.sc->chist[c][d] : 0u;
      s_cnt[c * kMaxRadix + d] = 0u;
      sum[c] += size[c][i];
    }
  }
  __syncthreads();
  // rank of each point among the tile's points of its row, in any order
  uint32_t rxy[kKpt], rz[kKpt];  // x row in the low, y row in the high half; z row
#pragma unroll
  for (int j = 0; j < kKpt; ++j) {
    rxy[j] = rz[j] = 0u;
    if (base + j * THREADS + tid < end) {
      const uint32_t rx = atomicAdd(&s_cnt[code[j] & m], 1u);
      const uint32_t ry = atomicAdd(&s_cnt[kMaxRadix + ((code[j] >> b) & m)], 1u);
      rz[j] = atomicAdd(&s_cnt[2 * kMaxRadix + (code[j] >> (2 * b))], 1u);
      rxy[j] = rx | (ry << 16);
    }
  }
  // the rows' starts in the frame
  uint32_t start[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const uint32_t x = warp_inclusive(sum[c], lane);
    if (lane == 31) s_w[c][warp] = x;
    start[c] = x - sum[c];
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 3; ++c) start[c] += warps_before(s_w[c], lane, warp);
  if (t == 0) {
    // for the sort: the rows' starts and the coordinates' extents
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      uint32_t s = start[c], lo = m, hi = 0u;
#pragma unroll
      for (int i = 0; i < kDpt; ++i) {
        const uint32_t d = uint32_t(tid * kDpt + i);
        if (int(d) < radix) a.sc->row_start[c][d] = s;
        s += size[c][i];
        if (size[c][i]) {
          lo = min(lo, d);
          hi = max(hi, d);
        }
      }
      if (tid == 0) a.sc->row_start[c][radix] = uint32_t(n);
      lo = __reduce_min_sync(0xffffffffu, lo);
      hi = __reduce_max_sync(0xffffffffu, hi);
      if (lane == 0) {
        // kept as maxima of (2^b - 1 - coordinate) and of the coordinate: zeroed with the build scalars
        atomicMax(&a.sc->row_ext[c][0], m - lo);
        atomicMax(&a.sc->row_ext[c][1], hi);
      }
    }
  }
  // reserve this tile's share of its rows, and the rows' starts inside the tile
  uint32_t cnt[3][kDpt], at[3][kDpt], own[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    own[c] = 0u;
#pragma unroll
    for (int i = 0; i < kDpt; ++i) {
      const int d = tid * kDpt + i;
      cnt[c][i] = s_cnt[c * kMaxRadix + d];
      at[c][i] = start[c] + (cnt[c][i] ? atomicAdd(&a.sc->row_used[c][d], cnt[c][i]) : 0u);
      start[c] += size[c][i];
      own[c] += cnt[c][i];
    }
    const uint32_t x = warp_inclusive(own[c], lane);
    if (lane == 31) s_w[3 + c][warp] = x;
    own[c] = x - own[c];
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    uint32_t s = own[c] + warps_before(s_w[3 + c], lane, warp);
#pragma unroll
    for (int i = 0; i < kDpt; ++i) {
      const int d = tid * kDpt + i;
      s_at[c * kMaxRadix + d] = s;
      s_cnt[c * kMaxRadix + d] = at[c][i] - s;  // + place in the tile = place in the frame
      s += cnt[c][i];
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int rc = row_coord(c);
#pragma unroll
    for (int j = 0; j < kKpt; ++j) {
      const int i = base + j * THREADS + tid;
      if (i < end) {
        const uint32_t k = code_from_c1(c, code[j], b, m);
        const uint32_t r = c == 0 ? rz[j] : c == 1 ? (rxy[j] & 0xffffu) : (rxy[j] >> 16);
        s_pt[s_at[rc * kMaxRadix + (k >> (2 * b))] + r] = make_uint2(uint32_t(i), k);
      }
    }
    __syncthreads();
    uint2* out = a.row_pts[c];
#pragma unroll
    for (int j = 0; j < kKpt; ++j) {
      const int p = j * THREADS + tid;
      if (p < end - base) {
        const uint2 e = s_pt[p];
        const uint32_t g = s_cnt[rc * kMaxRadix + (e.y >> (2 * b))] + uint32_t(p);
        if (g < uint32_t(n)) out[g] = e;
      }
    }
    if (c < 2) __syncthreads();
  }
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS, ScatterShape<THREADS>::kMinBlocks) k_bucket_scatter(BucketArgs a) {
  pdl_wait();
  bucket_scatter_body<THREADS>(a, blockIdx.x);
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS, ScatterShape<THREADS>::kMinBlocks)
    k_bucket_scatter_seg(const __grid_constant__ Seg<BucketArgs> s) {
  pdl_wait();
  const int f = seg_frame(s, blockIdx.x);
  bucket_scatter_body<THREADS>(s.a[f], blockIdx.x - s.start[f]);
}

// ---------------------------------------------------------------- order inside the rows
// One block per window of a.window output positions of a code.  It owns the
// rows of up to kRowMax points that start in the window, and of a larger row
// the lines (points of one second coordinate; their starts come from a
// histogram of the row) that start in it, so every point has one owner and an
// item holds at most window + kRowMax points unless one line repeats voxels
// thousands of times.  The points of rows above kRowSplit are put line by line first
// (next_split_window).  The item's points go into kSortBuckets buckets by the
// leading bits of their code (relative to the item's first row, and to the
// second coordinate's extent), and inside a bucket each point's place is the
// number of smaller (code, index) pairs.  Where that leaves many points in a bucket the
// buckets follow the rows instead (item_by_rows).  Items that repeated voxels crowd are
// ordered by a bitonic sort, those that do not fit through a bitmap (item_radix_sort).
// Measured (1M body points, b = 10): 38 us for the three codes, of which the
// prologue 7, counting 6, placing 5, ranking and writing 17; it is bound by its
// instructions (22 M a launch) and by the barriers between its phases.  With the
// row scatter it replaced three global radix passes and a slab sort: the graph's
// sorting launches took 112 us at 1M points and 54 us at 3k (12 launches), now 63
// and 17 (3 launches).  One counter a scan line in global memory instead (random
// atomics and writes in L2) took 110 us.  Windows of 1024 and 2048 positions were
// slower at 1M points (67 and 41 against 37 us: more prologues, and large rows are
// read by more blocks); splitting C1 from C2 and C3, to carry sorted ids, too (63).
constexpr int kBucketThreads = 1024;
constexpr int kRowMax = 7168;
constexpr int kWindowMax = 4096;
constexpr int kItemMax = kWindowMax + kRowMax;
constexpr int kSortBucketBits = 13;
constexpr int kSortBuckets = 1 << kSortBucketBits;  // 16-bit counters, two a word
constexpr uint32_t kBucketCoarse = 256;             // larger ones: the buckets follow the rows instead (item_by_rows)
constexpr size_t kBucketSmem = sizeof(uint2) * (size_t(kItemMax) + 4) + sizeof(uint16_t) * size_t(kSortBuckets);
static_assert(kSortBuckets == 8 * kBucketThreads && kMaxRadix <= kBucketThreads, "eight buckets, one row a thread");
static_assert(kItemMax < 65536, "16-bit places inside an item");

// Stable rank of one key among the equal digits of its warp (lanes in order),
// added to the warp's digit counter (16-bit half `half` of the pair word).
__device__ __forceinline__ uint32_t warp_rank(bool valid, uint32_t d, uint32_t* wh, int half, int lane) {
  const uint32_t peers = __match_any_sync(0xffffffffu, valid ? d : 0xffffffffu);
  const int leader = __ffs(peers) - 1;
  uint32_t old = 0;
  if (valid && lane == leader) old = (atomicAdd(&wh[d], uint32_t(__popc(peers)) << half) >> half) & 0xffffu;
  return __shfl_sync(0xffffffffu, old, leader) + __popc(peers & ((1u << lane) - 1u));
}

// A sorted point's outputs: code c, its place r, code k and input index idx.
__device__ __forceinline__ void emit_sorted(const BucketArgs& a, int c, uint32_t r, uint32_t k, uint32_t idx) {
  if (max(r, idx) >= uint32_t(a.n)) return;
  a.keys_out[c][r] = k;
  a.order_out[c][r] = int32_t(idx);
  if (c < 2) a.rank12[2 * size_t(idx) + c] = int32_t(r);
}

// An item as its slower paths take it.  Its points: its small rows, all of them side by
// side, and of up to two large rows the lines [mid0, mid1) that it owns, which take the
// places [line0, line1).  A split row's are at those places of row_tmp; of another row
// they are among all its points in row_pts.
struct ItemRows {
  const uint32_t* start;             // the code's row starts
  uint32_t ext0, ext1;               // the extent of the second coordinate
  uint32_t out0, total;              // the item's places
  uint32_t from, to;                 // the small rows
  uint32_t big[2];                   // 1 + the large row (0: none)
  uint32_t big_from[2], big_to[2];   // where its points are read
  uint32_t mid0[2], mid1[2], line0[2], line1[2];
  bool split[2];
};

// The points of an item that repeated voxels make too long or too crowded: into the
// order of their input indices, through a bitmap of the indices in shared memory, then by
// stable radix passes over the coordinates in which they differ (of the points of one voxel
// none), between row_tmp and the output arrays (the item's places).  One block, bound
// by its instructions and its scattered stores.  The graph of 100,000 points in one voxel
// takes 266 us, with radix passes over the index and all of the code 1410; of 20,000 beside
// a sphere of as many 234 and 330.  (Its steps are calls of their own: inlined,
// they cost the windows' sort its registers, 5 us at 1M points.)
constexpr int kRadixPer = 2;             // points a thread at a time
constexpr int kBitmapWords = 24 * 1024;  // input indices a time, 32 a word
static_assert(sizeof(uint32_t) * kBitmapWords <= kBucketSmem, "the bitmap fits the shared memory of an item");

// the digit of a code: its bits [shift, shift + bits)
struct Digit {
  int shift, bits;
  __device__ __forceinline__ uint32_t operator()(uint32_t code) const { return (code >> shift) & ((1u << bits) - 1u); }
};

// place i of an item in row_tmp (buf 0) or the output arrays (buf 1)
__device__ __forceinline__ uint2 radix_load(const BucketArgs& a, int c, uint32_t out0, int buf, uint32_t i) {
  i += out0;
  return buf == 0 ? __ldcg(a.row_tmp[c] + i) : make_uint2(uint32_t(__ldcg(a.order_out[c] + i)), __ldcg(a.keys_out[c] + i));
}
__device__ __forceinline__ void radix_store(const BucketArgs& a, int c, const ItemRows& rows, int buf, uint32_t i, uint2 e) {
  if (i >= rows.total) return;
  i += rows.out0;
  if (buf == 0) {
    a.row_tmp[c][i] = e;
  } else {
    a.keys_out[c][i] = e.y;
    a.order_out[c][i] = int32_t(e.x);
  }
}

// The item's points into the output arrays: its small rows at their places, of a large row
// the points on its lines at theirs, in any order; and the bits in which their codes differ.
template <bool SPLIT>
__device__ __noinline__ void radix_gather(const BucketArgs& a, int c, const ItemRows& rows, uint32_t* s_vary) {
  __shared__ uint32_t s_n;
  const int tid = threadIdx.x, lane = tid & 31;
  const int b = a.bits;
  const uint2* pts = a.row_pts[c];
#pragma unroll 4
  for (uint32_t i = rows.from + tid; i < rows.to; i += kBucketThreads) radix_store(a, c, rows, 1, i - rows.out0, pts[i]);
  for (int g = 0; g < 2; ++g) {
    const uint32_t to = rows.big_to[g];
    if (SPLIT && rows.split[g]) {
#pragma unroll 4
      for (uint32_t i = rows.big_from[g] + tid; i < to; i += kBucketThreads)
        radix_store(a, c, rows, 1, i - rows.out0, __ldcg(a.row_tmp[c] + i));
      continue;
    }
    if (tid == 0) s_n = rows.line0[g];
    __syncthreads();
    for (uint32_t i0 = rows.big_from[g] + uint32_t(tid & ~31); i0 < to; i0 += kBucketThreads) {
      const bool in = i0 + lane < to;
      const uint2 e = pts[in ? i0 + lane : i0];
      const uint32_t mid = (e.y >> b) & ((1u << b) - 1u);
      const bool own = in && mid >= rows.mid0[g] && mid < rows.mid1[g];
      const uint32_t who = __ballot_sync(0xffffffffu, own);
      uint32_t p = 0u;
      if (lane == 0 && who) p = atomicAdd(&s_n, uint32_t(__popc(who)));
      p = __shfl_sync(0xffffffffu, p, 0) + __popc(who & ((1u << lane) - 1u));
      if (own) radix_store(a, c, rows, 1, p - rows.out0, e);
    }
    __syncthreads();
  }
  if (tid == 0) *s_vary = 0u;
  __syncthreads();
  const uint32_t* keys = a.keys_out[c] + rows.out0;
  const uint32_t k0 = __ldcg(keys);
  uint32_t v = 0u;
#pragma unroll 4
  for (uint32_t i = tid; i < rows.total; i += kBucketThreads) v |= __ldcg(keys + i) ^ k0;
  v = __reduce_or_sync(0xffffffffu, v);
  if (lane == 0) atomicOr(s_vary, v);
  __syncthreads();
}

// words of the bitmap of the indices from i0 on
__device__ __forceinline__ uint32_t bitmap_words(int n, uint32_t i0) {
  return min((uint32_t(n) - i0 + 31u) / 32u, uint32_t(kBitmapWords));
}

// The input indices i0 .. i0 + 32 kBitmapWords - 1 of the item's points (in order_out) as a bitmap.
__device__ __noinline__ void fill_bitmap(const BucketArgs& a, int c, const ItemRows& rows, uint32_t i0, uint32_t* s_bits) {
  const uint32_t words = bitmap_words(a.n, i0);
  for (uint32_t i = threadIdx.x; i < words; i += kBucketThreads) s_bits[i] = 0u;
  __syncthreads();
  const int32_t* order = a.order_out[c] + rows.out0;
#pragma unroll 4
  for (uint32_t i = threadIdx.x; i < rows.total; i += kBucketThreads) {
    const uint32_t at = uint32_t(__ldcg(order + i)) - i0;
    if (at < 32u * words) atomicOr(&s_bits[at >> 5], 1u << (at & 31u));
  }
  __syncthreads();
}

// A bitmap's indices in ascending order into row_tmp, from the item's place `base` on; the place
// behind them.  A warp writes out a run of words, 32 bits of one word at a time.
__device__ __noinline__ uint32_t write_bitmap(const BucketArgs& a, int c, const ItemRows& rows, uint32_t i0, uint32_t base,
                                              const uint32_t* s_bits) {
  __shared__ uint32_t s_sw[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t words = bitmap_words(a.n, i0), run = (words + 31u) / 32u;  // of a warp
  const uint32_t from = min(words, warp * run), to = min(words, from + run);
  uint32_t mine = 0u;
  for (uint32_t i = from + lane; i < to; i += 32u) mine += __popc(s_bits[i]);
  mine = __reduce_add_sync(0xffffffffu, mine);
  if (lane == 0) s_sw[warp] = mine;
  __syncthreads();
  uint32_t p = base + warps_before(s_sw, lane, warp);
  for (uint32_t w0 = from; w0 < to; w0 += 32u) {
    const uint32_t word = w0 + lane < to ? s_bits[w0 + lane] : 0u;
    for (uint32_t todo = __ballot_sync(0xffffffffu, word != 0u); todo; todo &= todo - 1u) {
      const int l = __ffs(todo) - 1;
      const uint32_t w = __shfl_sync(0xffffffffu, word, l), at = p + __popc(w & ((1u << lane) - 1u));
      if (((w >> lane) & 1u) && at < rows.total) a.row_tmp[c][rows.out0 + at].x = i0 + 32u * (w0 + uint32_t(l)) + lane;
      p += __popc(w);
    }
  }
  base += __reduce_add_sync(0xffffffffu, s_sw[lane]);
  __syncthreads();
  return base;
}

// The points into row_tmp in the order of their input indices, with their codes.
__device__ __noinline__ void place_by_index(const BucketArgs& a, int c, const ItemRows& rows, uint32_t* s_bits) {
  uint32_t base = 0u;
  for (uint32_t i0 = 0u; i0 < uint32_t(a.n); i0 += 32u * kBitmapWords) {
    fill_bitmap(a, c, rows, i0, s_bits);
    base = write_bitmap(a, c, rows, i0, base, s_bits);
  }
  const uint32_t m = (1u << a.bits) - 1u;
  for (uint32_t i = threadIdx.x; i < rows.total; i += kBucketThreads) {
    uint2* e = a.row_tmp[c] + rows.out0 + i;
    const uint32_t idx = __ldcg(&e->x);
    if (idx >= uint32_t(a.n)) continue;
    const int32_t* q = a.xyz + 3 * size_t(idx);
    e->y = code_of(c, uint32_t(q[0]) & m, uint32_t(q[1]) & m, uint32_t(q[2]) & m, a.bits);
  }
  __syncthreads();
}

// Every digit's first place into s_run (points of one digit side by side are counted together).
__device__ __noinline__ void radix_count(const BucketArgs& a, int c, const ItemRows& rows, Digit digit, int cur,
                                         uint32_t* s_run) {
  __shared__ uint32_t s_sw[32];
  const int tid = threadIdx.x, lane = tid & 31;
  s_run[tid] = 0u;
  __syncthreads();
#pragma unroll 4
  for (uint32_t i0 = uint32_t(tid & ~31); i0 < rows.total; i0 += kBucketThreads) {
    const bool in = i0 + lane < rows.total;
    const uint32_t d = digit(radix_load(a, c, rows.out0, cur, in ? i0 + lane : i0).y);
    const uint32_t valid = __ballot_sync(0xffffffffu, in);
    if (__all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {
      if (lane == 0) atomicAdd(&s_run[d], uint32_t(__popc(valid)));
    } else if (in) {
      atomicAdd(&s_run[d], 1u);
    }
  }
  __syncthreads();
  const uint32_t run = block_exclusive(s_run[tid], s_sw);
  __syncthreads();
  s_run[tid] = run;
  __syncthreads();
}

// The points from buffer cur to their digits' places in the other, those of one digit in the
// order they have.
__device__ __noinline__ void radix_place(const BucketArgs& a, int c, const ItemRows& rows, Digit digit, int cur,
                                         uint32_t* smem) {
  constexpr int kPairs = kBucketThreads / 64;
  uint32_t* s_run = smem;                         // [kMaxRadix] each digit's next place
  uint32_t* s_at = s_run + kMaxRadix;             // [kMaxRadix] its first place among the points at hand
  uint32_t* s_cnt = s_at + kMaxRadix;             // [kPairs][kMaxRadix] two warps a word
  uint2* s_e = reinterpret_cast<uint2*>(s_cnt + kPairs * kMaxRadix);  // [kRadixPer][kBucketThreads] digit by digit
  static_assert(sizeof(uint32_t) * (kPairs + 2) * kMaxRadix + sizeof(uint2) * kRadixPer * kBucketThreads <= kBucketSmem,
                "they fit the shared memory of an item");
  __shared__ uint32_t s_sw[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* wh = s_cnt + (warp >> 1) * kMaxRadix;
  const int half = 16 * (warp & 1);
  for (uint32_t c0 = 0; c0 < rows.total; c0 += kRadixPer * kBucketThreads) {
    for (int i = tid; i < kPairs * kMaxRadix / 4; i += kBucketThreads)
      reinterpret_cast<uint4*>(s_cnt)[i] = make_uint4(0u, 0u, 0u, 0u);
    const uint32_t count = min(rows.total - c0, uint32_t(kRadixPer * kBucketThreads));
    const uint32_t pos = uint32_t(warp * 32 * kRadixPer + lane);  // a warp's points side by side
    uint2 e[kRadixPer];
    uint32_t rk[kRadixPer];
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j)
      e[j] = pos + 32u * j < count ? radix_load(a, c, rows.out0 + c0, cur, pos + 32u * j) : make_uint2(0u, 0u);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j) rk[j] = warp_rank(pos + 32u * j < count, digit(e[j].y), wh, half, lane);
    __syncthreads();
    // thread d: the warps' offsets of digit d, and the digit's points at hand
    uint32_t w0 = 0u;
#pragma unroll 4
    for (int w = 0; w < kPairs; ++w) {
      const uint32_t q = s_cnt[w * kMaxRadix + tid];
      s_cnt[w * kMaxRadix + tid] = w0 | ((w0 + (q & 0xffffu)) << 16);
      w0 += (q & 0xffffu) + (q >> 16);
    }
    s_at[tid] = block_exclusive(w0, s_sw);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j)
      if (pos + 32u * j < count) {
        const uint32_t d = digit(e[j].y);
        s_e[s_at[d] + ((wh[d] >> half) & 0xffffu) + rk[j]] = e[j];
      }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRadixPer; ++j) {
      const uint32_t p = uint32_t(j * kBucketThreads + tid);
      if (p < count) {
        const uint2 v = s_e[p];
        const uint32_t d = digit(v.y);
        radix_store(a, c, rows, cur ^ 1, s_run[d] + p - s_at[d], v);
      }
    }
    __syncthreads();
    s_run[tid] += w0;
  }
  __syncthreads();
}

template <bool SPLIT>
__device__ __noinline__ void item_radix_sort(const BucketArgs& a, int c, const ItemRows& rows, uint32_t* smem) {
  __shared__ uint32_t s_vary;
  radix_gather<SPLIT>(a, c, rows, &s_vary);
  place_by_index(a, c, rows, smem);
  int cur = 0;
  for (int f = 0; f < 3; ++f) {
    const Digit digit{a.bits * f, a.bits};
    if (digit(s_vary) == 0u) continue;
    radix_count(a, c, rows, digit, cur, smem);
    radix_place(a, c, rows, digit, cur, smem);
    cur ^= 1;
  }
  for (uint32_t i = threadIdx.x; i < rows.total; i += kBucketThreads) {
    const uint2 e = radix_load(a, c, rows.out0, cur, i);
    emit_sorted(a, c, rows.out0 + i, e.y, e.x);
  }
}

// A code's bucket: the leading bits of the code with the unused high bits of
// the second coordinate taken out (`base`: the first row and the smallest second
// coordinate; `gap` = 2^2b - 2^(b + bits of the second coordinate's extent)).
struct BucketOf {
  uint32_t base, gap;
  int row_shift, shift;
  __device__ __forceinline__ uint32_t operator()(uint32_t k) const {
    const uint32_t d = k - base;
    return min((d - (d >> row_shift) * gap) >> shift, uint32_t(kSortBuckets - 1));
  }
};

// for the rows [row0, row1] and second coordinates [mid0, mid1]
__device__ __forceinline__ BucketOf bucket_of(uint32_t row0, uint32_t row1, uint32_t mid0, uint32_t mid1, int b) {
  const int mid_bits = 32 - __clz(int(mid1 - mid0));
  BucketOf f;
  f.base = (row0 << (2 * b)) + (mid0 << b);
  f.gap = (1u << (2 * b)) - (1u << (b + mid_bits));
  f.row_shift = 2 * b;
  // the smallest shift that leaves at most kSortBuckets buckets
  f.shift = max(0, (32 - __clz(int(row1 - row0))) + mid_bits + b - kSortBucketBits);
  return f;
}

// adds one to bucket bk's counter (16 bits, two a word); its value before
__device__ __forceinline__ uint32_t count_in(uint32_t* s_cnt, uint32_t bk) {
  const uint32_t half = (bk & 1u) << 4;
  return (atomicAdd(&s_cnt[bk >> 1], 1u << half) >> half) & 0xffffu;
}

// The buckets' counters turned into their starts; returns this thread's largest count.
__device__ __forceinline__ uint32_t bucket_starts(uint32_t* s_cnt, uint32_t* s_w) {
  const int tid = threadIdx.x;
  uint32_t v[4] = {s_cnt[4 * tid], s_cnt[4 * tid + 1], s_cnt[4 * tid + 2], s_cnt[4 * tid + 3]};
  uint32_t sum = 0u, most = 0u;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    sum += (v[i] & 0xffffu) + (v[i] >> 16);
    most = max(most, max(v[i] & 0xffffu, v[i] >> 16));
  }
  uint32_t q = block_exclusive(sum, s_w);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t w = v[i];
    v[i] = q + ((q + (w & 0xffffu)) << 16);
    q += (w & 0xffffu) + (w >> 16);
  }
  reinterpret_cast<uint4*>(s_cnt)[tid] = make_uint4(v[0], v[1], v[2], v[3]);
  return most;
}

// The placed points of an item (four entries of padding behind them) to their places from out0.
template <typename Bucket>
__device__ __forceinline__ void rank_item(const BucketArgs& a, int c, const Bucket& bucket,
                                          const unsigned long long* s_pt, const uint32_t* s_cnt, uint32_t out0,
                                          uint32_t total) {
  // counter k is now the end of bucket k.  The points before a bucket are
  // smaller and those behind it larger, so the counting may start at a
  // multiple of four and run past the end: four points a step, no tail.
  const uint16_t* s_end = reinterpret_cast<const uint16_t*>(s_cnt);  // bucket k's counter
  for (uint32_t p = threadIdx.x; p < total; p += kBucketThreads) {
    const unsigned long long me = s_pt[p];
    const uint32_t k = uint32_t(me >> 32), bk = bucket(k);
    const uint32_t first = (bk ? uint32_t(s_end[bk - 1]) : 0u) & ~3u, last = min(uint32_t(s_end[bk]), total);
    uint32_t r = out0 + first;
#pragma unroll 1
    for (uint32_t j = first; j < last; j += 4) {
      const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(s_pt + j);
      const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(s_pt + j + 2);
      r += (u.x < me) + (u.y < me) + (w.x < me) + (w.y < me);
    }
    emit_sorted(a, c, r, k, uint32_t(me));
  }
}

// Buckets that follow the item's rows: a row has as many of them as points, over the
// second coordinate's extent (a large row over the item's lines), so they stay small where
// the rows lie far apart (two bodies, one above the other) or a few stray points make
// the extent many times that of the rest.
struct BucketByRow {
  const ItemRows& it;
  int b, n;
  uint32_t scale;  // buckets a place, 2^-16
  __device__ __forceinline__ uint32_t operator()(uint32_t k) const {
    const uint32_t m = (1u << b) - 1u, row = k >> (2 * b);
    uint32_t at = it.start[row], end = min(it.start[row + 1], uint32_t(n)), mid0 = it.ext0, span = it.ext1 - it.ext0;
#pragma unroll
    for (int g = 0; g < 2; ++g)
      if (row + 1u == it.big[g]) {
        at = it.line0[g];
        end = it.line1[g];
        mid0 = it.mid0[g];
        span = it.mid1[g] - 1u - mid0;
      }
    const uint32_t in_row = ((((k >> b) & m) - mid0) << b) | (k & m);
    const int bits = 32 - __clz(int(span)) + b;
    const uint32_t place = at - it.out0 + uint32_t(((unsigned long long)(end - at) * in_row) >> bits);
    return min(uint32_t(((unsigned long long)place * scale) >> 16), uint32_t(kSortBuckets - 1));
  }
};

// The item's points in s_pt by a bitonic sort of (code, index), in the form whose merges begin
// with mirrored pairs, so that every exchange is ascending and places behind the last
// point need not exist.  A warp's pairs of up to 64 places lie in 64 places of its own.
__device__ __noinline__ void bitonic_item(unsigned long long* s_pt, uint32_t total) {
  const uint32_t tid = threadIdx.x;
  const auto exchange = [&](uint32_t lo, uint32_t hi) {
    if (hi >= total) return;
    const unsigned long long x = s_pt[lo], y = s_pt[hi];
    if (y < x) {
      s_pt[lo] = y;
      s_pt[hi] = x;
    }
  };
  const int top = 32 - __clz(int(total - 1u));  // 2^top places hold the points
  const uint32_t pairs = total > 1u ? 1u << (top - 1) : 0u;
  for (int k = 1; k <= top; ++k) {
    // blocks of 2^k places: mirrored pairs, then pairs 2^j apart
    if (k > 6) __syncthreads();
    for (uint32_t t = tid; t < pairs; t += kBucketThreads) {
      const uint32_t in = t & ((1u << (k - 1)) - 1u), at = (t >> (k - 1)) << k;
      exchange(at + in, at + (1u << k) - 1u - in);
    }
    int j = k - 2;
    for (; j > 5; --j) {
      __syncthreads();
      for (uint32_t t = tid; t < pairs; t += kBucketThreads) {
        const uint32_t lo = ((t >> j) << (j + 1)) + (t & ((1u << j) - 1u));
        exchange(lo, lo + (1u << j));
      }
    }
    if (k > 6) __syncthreads();
    for (; j >= 0; --j) {
      __syncwarp();
      for (uint32_t t = tid; t < pairs; t += kBucketThreads) {
        const uint32_t lo = ((t >> j) << (j + 1)) + (t & ((1u << j) - 1u));
        exchange(lo, lo + (1u << j));
      }
    }
    __syncwarp();
  }
  __syncthreads();
}

// An item whose buckets were too large: with buckets that follow its rows; what is then
// still crowded, by repeated voxels, through the bitonic sort or, where the points differ in
// one coordinate at most, through the bitmap (5,000 points in one voxel: the graph 39 us, by
// the bitonic sort 74); and an item that does not fit, through the bitmap.
// (Two spheres of 200,000 points apart along an axis: the sort 84 us with the items across
// the gap by a radix sort, 22 so; a block of 20^3 voxels and two points in the grid's
// corners: the graph 90 -> 39.)  Counting a second time pays from buckets of some 256
// points on: a box surface of 300,000 points, whose edges fill buckets of 256, 97 us, with
// a limit of 128 108; a sphere of 100,000 points with two stray ones 43 and 35.  The
// bitonic sort takes the place of a point's comparisons with more than kCrowded others on
// average: the graph of 2,000 voxels 500 times each takes 314 us, with comparisons 458; of
// 4,096 voxels 244 times each 450 and 347.
constexpr uint32_t kCrowded = 320;
template <bool SPLIT>
__device__ __noinline__ void item_by_rows(const BucketArgs& a, int c, const ItemRows& rows, uint32_t* smem) {
  if (rows.total > uint32_t(kItemMax)) {
    item_radix_sort<SPLIT>(a, c, rows, smem);
    return;
  }
  unsigned long long* s_pt = reinterpret_cast<unsigned long long*>(smem);
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_pt + kItemMax + 4);
  __shared__ uint32_t s_w[32], s_sq, s_and, s_or;
  const int tid = threadIdx.x, b = a.bits;
  const uint32_t m = (1u << b) - 1u;
  const BucketByRow bucket{rows, b, a.n, (uint32_t(kSortBuckets) << 16) / rows.total};
  const auto points = [&](auto&& f) {
    for (uint32_t i = rows.from + tid; i < rows.to; i += kBucketThreads) f(a.row_pts[c][i]);
    for (int g = 0; g < 2; ++g)
      for (uint32_t i = rows.big_from[g] + tid; i < rows.big_to[g]; i += kBucketThreads) {
        const uint2 e = SPLIT && rows.split[g] ? __ldcg(a.row_tmp[c] + i) : a.row_pts[c][i];
        const uint32_t mid = (e.y >> b) & m;
        if (mid >= rows.mid0[g] && mid < rows.mid1[g]) f(e);
      }
  };
  __syncthreads();
  reinterpret_cast<uint4*>(s_cnt)[tid] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    s_sq = s_or = 0u;
    s_and = ~0u;
  }
  __syncthreads();
  uint32_t all = ~0u, any = 0u;  // the bits that all, and any of the codes have
  points([&](uint2 e) {
    count_in(s_cnt, bucket(e.y));
    all &= e.y;
    any |= e.y;
  });
  all = __reduce_and_sync(0xffffffffu, all);
  any = __reduce_or_sync(0xffffffffu, any);
  if ((tid & 31) == 0) {
    atomicAnd(&s_and, all);
    atomicOr(&s_or, any);
  }
  __syncthreads();
  // the comparisons that ranking would make (at most kItemMax squared, below 2^27)
  uint32_t sq = 0u;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t w = s_cnt[4 * tid + i];
    sq += (w & 0xffffu) * (w & 0xffffu) + (w >> 16) * (w >> 16);
  }
  sq = __reduce_add_sync(0xffffffffu, sq);
  if ((tid & 31) == 0) atomicAdd(&s_sq, sq);
  bucket_starts(s_cnt, s_w);
  __syncthreads();
  points([&](uint2 e) {
    const uint32_t p = count_in(s_cnt, bucket(e.y));
    if (p < uint32_t(kItemMax)) s_pt[p] = ((unsigned long long)e.y << 32) | e.x;
  });
  if (tid < 4) s_pt[rows.total + tid] = ~0ull;
  __syncthreads();
  if (s_sq <= kCrowded * rows.total) {
    rank_item(a, c, bucket, s_pt, s_cnt, rows.out0, rows.total);
    return;
  }
  const uint32_t vary = s_and ^ s_or;
  if (((vary & m) != 0u) + (((vary >> b) & m) != 0u) + (vary >> (2 * b) != 0u) < 2) {
    item_radix_sort<SPLIT>(a, c, rows, smem);
    return;
  }
  bitonic_item(s_pt, rows.total);
  for (uint32_t i = tid; i < rows.total; i += kBucketThreads)
    emit_sorted(a, c, rows.out0 + i, uint32_t(s_pt[i] >> 32), uint32_t(s_pt[i]));
}

// the line counters of code c's split row that starts at place `first`
__device__ __forceinline__ uint32_t* line_counters(const BucketArgs& a, int c, uint32_t first) {
  return a.lines + (size_t(c) * size_t(a.line_slots) + first / uint32_t(kRowSplit + 1)) * size_t(2 * kMaxRadix);
}

// One window of a code.  SPLIT: the code has rows above kRowSplit points, which lie line by
// line in row_tmp, the points of every line counted; false (and nothing done) if it has
// such rows and they do not.
enum class Window { kDone, kHasSplitRows, kCrowded };
template <bool SPLIT>
__device__ __forceinline__ Window sort_window(const BucketArgs& a, int item, int c, ItemRows& s_rows) {
  const uint32_t* start = a.sc->row_start[row_coord(c)];
  extern __shared__ __align__(16) uint32_t smem[];
  // (code in the high, index in the low half; four entries of padding for the ranking loads)
  unsigned long long* s_pt = reinterpret_cast<unsigned long long*>(smem);     // [kItemMax + 4]
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_pt + kItemMax + 4);         // [kSortBuckets / 2]
  __shared__ uint32_t s_w[3][32];
  __shared__ uint32_t s_lo, s_hi, s_row0, s_row1;  // the small rows' places, the first and the last row
  __shared__ uint32_t s_big[2];                    // 1 + the large row that starts before / in the window
  __shared__ uint32_t s_mid0, s_mid1;              // a large row's own lines [mid0, mid1)
  __shared__ uint32_t s_first[2], s_last[2];       // and the places they take
  const int tid = threadIdx.x, lane = tid & 31;
  const int b = a.bits, radix = 1 << b, n = a.n;
  const uint32_t m = uint32_t(radix) - 1u;
  const DevScalars* sc = a.sc;
  const uint2* pts = a.row_pts[c];
  const uint32_t w0 = uint32_t(item) * uint32_t(a.window), w1 = w0 + uint32_t(a.window);
  const uint32_t rs = tid < radix ? start[tid] : 0u, re = tid < radix ? min(start[tid + 1], uint32_t(n)) : 0u;
  const int mc = mid_coord(c);
  reinterpret_cast<uint4*>(s_cnt)[tid] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    s_lo = s_row0 = s_first[0] = s_first[1] = 0xffffffffu;
    s_hi = s_row1 = s_big[0] = s_big[1] = s_last[0] = s_last[1] = 0u;
  }
  if (SPLIT) __syncthreads();
  else if (__syncthreads_or(re > rs && re - rs > uint32_t(kRowSplit))) return Window::kHasSplitRows;
  {
    uint32_t lo = 0xffffffffu, hi = 0u, row = 0xffffffffu;
    if (re > rs) {
      if (re - rs <= uint32_t(kRowMax)) {
        if (rs >= w0 && rs < w1) {
          lo = rs;
          hi = re;
          row = uint32_t(tid);
        }
      } else if (rs < w1 && re > w0) {
        s_big[rs < w0 ? 0 : 1] = uint32_t(tid) + 1u;
        row = uint32_t(tid);
      }
    }
    if (__any_sync(0xffffffffu, row != 0xffffffffu)) {
      lo = __reduce_min_sync(0xffffffffu, lo);
      hi = __reduce_max_sync(0xffffffffu, hi);
      const uint32_t r0 = __reduce_min_sync(0xffffffffu, row);
      const uint32_t r1 = __reduce_max_sync(0xffffffffu, row == 0xffffffffu ? 0u : row);
      if (lane == 0) {
        atomicMin(&s_lo, lo);
        atomicMax(&s_hi, hi);
        atomicMin(&s_row0, r0);
        atomicMax(&s_row1, r1);
      }
    }
  }
  __syncthreads();
  // the small rows lie side by side: [lo, lo + cnt_small), lo = 0 if there are none
  const uint32_t lo = s_hi ? s_lo : 0u, cnt_small = s_hi - lo;
  const uint32_t big[2] = {s_big[0], s_big[1]};
  if (!cnt_small && !big[0] && !big[1]) return Window::kDone;
  uint32_t out0 = cnt_small ? lo : 0xffffffffu, out1 = s_hi;  // the item's places [out0, out1)
  // large rows: where their points are read (split ones: the own lines' places), own lines
  uint32_t b0[2] = {0u, 0u}, b1[2] = {0u, 0u}, l0[2] = {0u, 0u}, l1[2] = {0u, 0u};
  bool split[2] = {false, false};
  if (big[0] | big[1]) {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      if (!big[g]) continue;
      b0[g] = start[big[g] - 1u];
      b1[g] = min(start[big[g]], uint32_t(n));
      if (SPLIT) split[g] = b1[g] - b0[g] > uint32_t(kRowSplit);
      if (tid == 0) {
        s_mid0 = 0xffffffffu;
        s_mid1 = 0u;
      }
      uint32_t v;  // the points of line tid
      if (SPLIT && split[g]) {
        __syncthreads();
        v = __ldcg(line_counters(a, c, b0[g]) + tid);
      } else {
        // the row's line histogram
#pragma unroll 4
        for (uint32_t i = b0[g] + tid; i < b1[g]; i += kBucketThreads) atomicAdd(&s_cnt[(pts[i].y >> b) & m], 1u);
        __syncthreads();
        v = s_cnt[tid];
      }
      // and the lines that start in the window
      const uint32_t at = b0[g] + block_exclusive(v, s_w[g]);
      s_cnt[tid] = 0u;
      const bool own = v && at >= w0 && at < w1;
      const uint32_t lo_w = __reduce_min_sync(0xffffffffu, own ? uint32_t(tid) : 0xffffffffu);
      const uint32_t hi_w = __reduce_max_sync(0xffffffffu, own ? uint32_t(tid) + 1u : 0u);
      if (lane == 0 && hi_w) {
        atomicMin(&s_mid0, lo_w);
        atomicMax(&s_mid1, hi_w);
      }
      if (own) {
        atomicMin(&s_first[g], at);
        atomicMax(&s_last[g], min(at + v, uint32_t(n)));
      }
      __syncthreads();
      l0[g] = s_mid0;
      l1[g] = s_mid1;
      if (SPLIT && split[g]) {
        b0[g] = min(s_first[g], uint32_t(n));
        b1[g] = s_last[g];
      }
      __syncthreads();
    }
    out0 = min(out0, min(s_first[0], s_first[1]));
    out1 = max(out1, max(s_last[0], s_last[1]));
    if (out0 >= out1) return Window::kDone;  // one long line crosses the window
  }
  const uint32_t total = out1 - out0;
  uint32_t mid0 = m - sc->row_ext[mc][0], mid1 = sc->row_ext[mc][1];
  if (s_row0 == s_row1 && (l1[0] | l1[1])) {
    // a part of one row: its buckets share out the own lines only
    mid0 = l1[0] ? l0[0] : l0[1];
    mid1 = (l1[0] ? l1[0] : l1[1]) - 1u;
  }
  const BucketOf bucket = bucket_of(s_row0, s_row1, mid0, mid1, b);
  const auto owned = [&](int g, uint32_t k) {
    const uint32_t mid = (k >> b) & m;
    return mid >= l0[g] && mid < l1[g];
  };
  const auto count = [&](uint32_t k) { return count_in(s_cnt, bucket(k)); };
  bool fits = total <= uint32_t(kItemMax);
  if (fits) {
#pragma unroll 4
    for (uint32_t i = lo + tid; i < lo + cnt_small; i += kBucketThreads) count(pts[i].y);
#pragma unroll
    for (int g = 0; g < 2; ++g)
      if (l1[g])
#pragma unroll 4
        for (uint32_t i = b0[g] + tid; i < b1[g]; i += kBucketThreads) {
          const uint32_t k = (SPLIT && split[g] ? __ldcg(a.row_tmp[c] + i) : pts[i]).y;
          if (owned(g, k)) count(k);
        }
    __syncthreads();
    fits = !__syncthreads_or(bucket_starts(s_cnt, s_w[2]) > kBucketCoarse);
  }
  if (!fits) {
    // (through shared memory: nothing of the loops around is kept on the stack for this)
    if (tid == 0) {
      s_rows.start = start;
      s_rows.ext0 = m - sc->row_ext[mc][0];
      s_rows.ext1 = sc->row_ext[mc][1];
      s_rows.out0 = out0;
      s_rows.total = total;
      s_rows.from = lo;
      s_rows.to = lo + cnt_small;
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        s_rows.big_from[g] = b0[g];
        s_rows.big_to[g] = l1[g] ? b1[g] : 0u;
        s_rows.mid0[g] = l0[g];
        s_rows.mid1[g] = l1[g];
        s_rows.big[g] = l1[g] ? s_big[g] : 0u;
        s_rows.line0[g] = s_first[g];
        s_rows.line1[g] = s_last[g];
        if (SPLIT) s_rows.split[g] = split[g];
      }
    }
    __syncthreads();
    return Window::kCrowded;
  }
  const auto put = [&](uint2 e) {
    const uint32_t p = count(e.y);
    if (p < uint32_t(kItemMax)) s_pt[p] = ((unsigned long long)e.y << 32) | e.x;
  };
#pragma unroll 4
  for (uint32_t i = lo + tid; i < lo + cnt_small; i += kBucketThreads) put(pts[i]);
#pragma unroll
  for (int g = 0; g < 2; ++g)
    if (l1[g])
#pragma unroll 4
      for (uint32_t i = b0[g] + tid; i < b1[g]; i += kBucketThreads) {
        const uint2 e = SPLIT && split[g] ? __ldcg(a.row_tmp[c] + i) : pts[i];
        if (owned(g, e.y)) put(e);
      }
  if (tid < 4) s_pt[total + tid] = ~0ull;
  __syncthreads();
  rank_item(a, c, bucket, s_pt, s_cnt, out0, total);
  return Window::kDone;
}

// Thread 0 waits until *counter reaches `target` (a bounded wait); false for every thread if it gave up.
__device__ __forceinline__ bool wait_count(const BucketArgs& a, const uint32_t* counter, uint32_t target, int* s_ok) {
  if (threadIdx.x == 0) {
    const unsigned long long t0 = global_ns(), limit = a.sc->wait_limit_ns;
    int ok = 1;
    while (ld_acquire_u32(counter) < target) {
      if (global_ns() - t0 > limit) {
        atomicOr(&a.sc->status, kFlagTimeout);
        ok = 0;
        break;
      }
      __nanosleep(64);
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// what this block's threads have written, published as `add` on *counter
__device__ __forceinline__ void publish_count(uint32_t* counter, uint32_t add) {
  __syncthreads();
  if (threadIdx.x == 0 && add) {
    __threadfence();
    atomicAdd(counter, add);
  }
}

// A code with rows above kRowSplit points (walls and floors along an axis).  Left as they
// are, every window of such a row reads the whole row three times to find its own lines,
// and the graph of a plane of 1M points took 580 us.  Instead the row's points are counted
// by line and put line by line into row_tmp, a window's positions at a time, before the
// windows are sorted: 115-120 us (91 for a sphere of 1M points).  The rows are split from
// 32768 points on because the three steps before the sort cost 20-40 us: rows of 8,000 and
// 10,000 points (1M in all) 110 and 122 us as they are, 169 and 181 split; of 31,000 160 and
// 165; of 100,000 (800,000 in all) 164 as they are, 115 split.
// The code's blocks take tickets: first the rows' counters are cleared, then the windows'
// points counted, then placed, then the windows sorted.  A block waits only for parts whose
// tickets were drawn before its own, that is by blocks already running, and those wait only
// for still earlier ones: whatever number of blocks is resident, the waits end.  (A launch
// of its own between the row scatter and the sort would cost frames without such rows
// 2-3 us.  All three codes' windows by common tickets, plain ones between the steps: 10 us
// slower than with the other codes' blocks beside them.)

// The next window to sort, or -1: none is left, or a wait gave up.
__device__ __noinline__ int next_split_window(const BucketArgs& a, int c) {
  const int items = (a.n + a.window - 1) / a.window;  // (the code's blocks)
  const uint32_t* start = a.sc->row_start[row_coord(c)];
  extern __shared__ __align__(16) uint32_t smem[];
  uint32_t* s_n = smem;                 // [kMaxRadix] this window's points of a line
  uint32_t* s_at = s_n + kMaxRadix;     // [kMaxRadix] and their first place
  __shared__ uint32_t s_big[2], s_ticket, s_rows, s_points, s_scan[32];
  __shared__ int s_ok;
  const int tid = threadIdx.x;
  const int b = a.bits, n = a.n;
  const uint32_t m = (1u << b) - 1u;
  DevScalars* sc = a.sc;
  // the row of this thread, if it is split
  const uint32_t rs = tid <= int(m) ? start[tid] : 0u, re = tid <= int(m) ? min(start[tid + 1], uint32_t(n)) : 0u;
  const bool mine = re > rs && re - rs > uint32_t(kRowSplit);
  if (tid == 0) s_rows = s_points = 0u;
  __syncthreads();
  if (mine) {
    atomicAdd(&s_rows, 1u);
    atomicAdd(&s_points, re - rs);
  }
  __syncthreads();
  const uint32_t rows = s_rows, points = s_points;
  for (;;) {
    __syncthreads();
    if (tid == 0) s_ticket = atomicAdd(&sc->sort_ticket[c], 1u);
    if (tid < 2) s_big[tid] = 0u;
    __syncthreads();
    const uint32_t phase = s_ticket / uint32_t(items), item = s_ticket % uint32_t(items);
    if (phase >= 3u)
      return phase == 3u && wait_count(a, &sc->lines_placed[c], points, &s_ok) ? int(item) : -1;
    // the split rows that overlap the window: 1 + the one that starts before it, and in it
    const uint32_t w0 = item * uint32_t(a.window), w1 = w0 + uint32_t(a.window);
    if (mine && rs < w1 && re > w0) s_big[rs < w0 ? 0 : 1] = uint32_t(tid) + 1u;
    __syncthreads();
    if (phase == 0u) {
      if (s_big[1]) {
        uint32_t* cnt = line_counters(a, c, start[s_big[1] - 1u]);
        for (int i = tid; i < 2 * kMaxRadix; i += kBucketThreads) cnt[i] = 0u;
      }
      publish_count(&sc->rows_cleared[c], s_big[1] ? 1u : 0u);
      continue;
    }
    if (phase == 1u ? !wait_count(a, &sc->rows_cleared[c], rows, &s_ok)
                    : !wait_count(a, &sc->lines_counted[c], points, &s_ok))
      return -1;
    uint32_t done = 0u;
    for (int g = 0; g < 2; ++g) {
      if (!s_big[g]) continue;
      const uint32_t first = start[s_big[g] - 1u];
      const uint32_t from = max(first, w0), to = min(min(start[s_big[g]], uint32_t(n)), w1);
      uint32_t* cnt = line_counters(a, c, first);
      const uint2* pts = a.row_pts[c];
      static_assert(kWindowMax <= 4 * kBucketThreads && kMaxRadix == kBucketThreads, "four points, one line a thread");
      s_n[tid] = 0u;
      __syncthreads();
      uint2 e[4];
      uint32_t r[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t i = from + uint32_t(j * kBucketThreads + tid);
        e[j] = i < to ? pts[i] : make_uint2(0u, 0u);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (from + uint32_t(j * kBucketThreads + tid) < to) r[j] = atomicAdd(&s_n[(e[j].y >> b) & m], 1u);
      __syncthreads();
      const uint32_t v = s_n[tid];
      if (phase == 1u) {
        if (v) atomicAdd(cnt + tid, v);
      } else {
        const uint32_t at = first + block_exclusive(__ldcg(cnt + tid), s_scan);
        s_at[tid] = v ? at + atomicAdd(cnt + kMaxRadix + tid, v) : 0u;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (from + uint32_t(j * kBucketThreads + tid) < to) {
            const uint32_t p = s_at[(e[j].y >> b) & m] + r[j];
            if (p < uint32_t(n)) a.row_tmp[c][p] = e[j];
          }
      }
      done += to > from ? to - from : 0u;
      __syncthreads();
    }
    publish_count(phase == 1u ? &sc->lines_counted[c] : &sc->lines_placed[c], done);
  }
}

// (calls of their own: inlined, they cost the other frames' sort its registers: 5 us at 1M points)
__device__ __noinline__ void sort_split_window(const BucketArgs& a, int item, int c) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ ItemRows s_rows;
  if (sort_window<true>(a, item, c, s_rows) == Window::kCrowded) item_by_rows<true>(a, c, s_rows, smem);
}

__device__ __noinline__ void sort_split_rows(const BucketArgs& a, int c) {
  for (;;) {
    const int item = next_split_window(a, c);
    if (item < 0) return;
    sort_split_window(a, item, c);
  }
}

// one block for every window of a code
__device__ __forceinline__ void bucket_sort_body(const BucketArgs& a, int block, int c) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ ItemRows s_rows;
  const Window w = sort_window<false>(a, block, c, s_rows);
  if (w == Window::kCrowded) item_by_rows<false>(a, c, s_rows, smem);
  else if (w == Window::kHasSplitRows) sort_split_rows(a, c);
}

__global__ void __launch_bounds__(kBucketThreads, 2) k_bucket_sort(const __grid_constant__ BucketArgs a) {
  pdl_wait();
  bucket_sort_body(a, blockIdx.x, blockIdx.y);
}

// A frame of up to kDirectMax points: the whole frame is one item of each code, so
// three blocks sort it from the coordinates, without histogram and row scatter;
// the other blocks zero the build's scalars, which nothing here reads.  A block
// takes eight points a thread (their codes stay in registers).  A frame of 2,000 points
// takes 57.5 us instead of 63.6, one of 8,192 63.6 instead of 65.6 (three launches fewer).
constexpr int kDirectPer = kDirectMax / kBucketThreads;
static_assert(kDirectMax <= kItemMax && kDirectPer * kBucketThreads == kDirectMax, "one item, whole points a thread");

__global__ void __launch_bounds__(kBucketThreads, 1) k_direct_sort(const __grid_constant__ BucketArgs a, ZeroArgs z) {
  pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31;
  if (blockIdx.x >= 3) {
    for (size_t i = size_t(blockIdx.x - 3) * kBucketThreads + tid; i < z.words; i += size_t(gridDim.x - 3) * kBucketThreads)
      z.p[i] = 0u;
    return;
  }
  extern __shared__ __align__(16) uint32_t smem[];
  unsigned long long* s_pt = reinterpret_cast<unsigned long long*>(smem);
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_pt + kItemMax + 4);
  __shared__ uint32_t s_w[32];
  __shared__ uint32_t s_lo[2], s_hi[2];  // smallest and largest row and second coordinate
  const int c = blockIdx.x, b = a.bits, n = a.n;
  const uint32_t m = (1u << b) - 1u;
  reinterpret_cast<uint4*>(s_cnt)[tid] = make_uint4(0u, 0u, 0u, 0u);
  if (tid < 2) {
    s_lo[tid] = 0xffffffffu;
    s_hi[tid] = 0u;
  }
  uint32_t x[kDirectPer], y[kDirectPer], zc[kDirectPer], code[kDirectPer];
#pragma unroll
  for (int j = 0; j < kDirectPer; ++j) {
    const int i = j * kBucketThreads + tid;
    x[j] = y[j] = zc[j] = 0u;
    if (i < n) {
      x[j] = uint32_t(a.xyz[3 * size_t(i)]);
      y[j] = uint32_t(a.xyz[3 * size_t(i) + 1]);
      zc[j] = uint32_t(a.xyz[3 * size_t(i) + 2]);
    }
  }
  __syncthreads();
  {
    bool bad = false;
    uint32_t r0 = 0xffffffffu, r1 = 0u, m0 = 0xffffffffu, m1 = 0u;
#pragma unroll
    for (int j = 0; j < kDirectPer; ++j) {
      bad |= (x[j] > m) | (y[j] > m) | (zc[j] > m);
      code[j] = code_of(c, x[j] & m, y[j] & m, zc[j] & m, b);
      if (j * kBucketThreads + tid < n) {
        const uint32_t row = code[j] >> (2 * b), mid = (code[j] >> b) & m;
        r0 = min(r0, row);
        r1 = max(r1, row);
        m0 = min(m0, mid);
        m1 = max(m1, mid);
      }
    }
    if (bad) atomicOr(&a.sc->status, kFlagRange);
    r0 = __reduce_min_sync(0xffffffffu, r0);
    r1 = __reduce_max_sync(0xffffffffu, r1);
    m0 = __reduce_min_sync(0xffffffffu, m0);
    m1 = __reduce_max_sync(0xffffffffu, m1);
    if (lane == 0) {
      atomicMin(&s_lo[0], r0);
      atomicMax(&s_hi[0], r1);
      atomicMin(&s_lo[1], m0);
      atomicMax(&s_hi[1], m1);
    }
  }
  __syncthreads();
  const BucketOf bucket = bucket_of(s_lo[0], s_hi[0], s_lo[1], s_hi[1], b);
#pragma unroll
  for (int j = 0; j < kDirectPer; ++j)
    if (j * kBucketThreads + tid < n) count_in(s_cnt, bucket(code[j]));
  __syncthreads();
  const uint32_t most = bucket_starts(s_cnt, s_w);
  if (__syncthreads_or(most > kBucketCoarse)) {
    // (item_by_rows reads the points and the row starts as the row scatter leaves them)
    __shared__ uint32_t s_start[kMaxRadix + 1];
    __shared__ ItemRows s_all;
    s_start[tid] = 0u;
    if (tid == 0) {
      s_start[kMaxRadix] = uint32_t(n);
      s_all = ItemRows{s_start, s_lo[1], s_hi[1], 0u, uint32_t(n), 0u, uint32_t(n)};
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kDirectPer; ++j) {
      const int i = j * kBucketThreads + tid;
      if (i < n) {
        a.row_pts[c][i] = make_uint2(uint32_t(i), code[j]);
        atomicAdd(&s_start[code[j] >> (2 * b)], 1u);
      }
    }
    __syncthreads();
    const uint32_t first = block_exclusive(s_start[tid], s_w);
    __syncthreads();
    s_start[tid] = first;
    __syncthreads();
    item_by_rows<false>(a, c, s_all, smem);
    return;
  }
#pragma unroll
  for (int j = 0; j < kDirectPer; ++j) {
    const int i = j * kBucketThreads + tid;
    if (i < n) {
      const uint32_t p = count_in(s_cnt, bucket(code[j]));
      if (p < uint32_t(kItemMax)) s_pt[p] = ((unsigned long long)code[j] << 32) | uint32_t(i);
    }
  }
  if (tid < 4) s_pt[n + tid] = ~0ull;
  __syncthreads();
  rank_item(a, c, bucket, s_pt, s_cnt, 0u, uint32_t(n));
}

// segmented: frame f's blocks are runs of equal length, one per code
__global__ void __launch_bounds__(kBucketThreads, 2) k_bucket_sort_seg(const __grid_constant__ Seg<BucketArgs> s) {
  pdl_wait();
  const int f = seg_frame(s, blockIdx.x);
  const int local = blockIdx.x - s.start[f], items = (s.start[f + 1] - s.start[f]) / 3;
  bucket_sort_body(s.a[f], local % items, local / items);
}

// One code's order per group of gx blocks (block x of code c).  Code 0 is the C1 order
// itself; codes 1 and 2 read the input indices along C2 and C3 and the codes in
// the same order (code c's own packing; a distance does not depend on it) and
// gather each point's sorted id and, beside it, its C2 rank by input index (one
// array of pairs: 27.8 us at 1M points, 29.4 with two arrays).  The two million
// random reads and the slot writes bound it (6.8 M L2 sectors).  Each lane takes four consecutive positions
// (16-byte loads, the gathers issued together); the neighbours across lanes
// come from shuffles, with one extra lookup at each end of the warp.  With
// colours (a whole run), the blocks of code 0, which have no slots to write, also
// take the colours into the C1 order (colors_quad): 29.8 us with them, against
// 9.7 us for a launch of its own.
struct LinkPt {
  int k;       // sorted (C1) id, -1 outside [0, n)
  int r2;      // position in the C2 order (code 2 only)
  uint32_t c;  // packed code of the order
};

// the sorted id (x) and the C2 rank (y, code 2 only) of the point at position r of
// a code; x = -1 outside the frame
__device__ __forceinline__ int2 link_id(int r, int n, int code, const int32_t* __restrict__ ord,
                                        const int2* __restrict__ rank12) {
  if (code == 0) return make_int2(r, -1);
  const int i = ord[r];
  if (!in_range(i, n)) return make_int2(-1, -1);
  int2 q = make_int2(-1, -1);
  if (code == 1) q.x = rank12[i].x;
  else q = rank12[i];
  if (!in_range(q.x, n)) q.x = -1;
  return q;
}

// a packed code of order c as a C1 code
__device__ __forceinline__ uint32_t c1_from_code(int c, uint32_t k, int b) {
  const uint32_t m = (1u << b) - 1u;
  const uint32_t hi = (k >> (2 * b)) & m, mid = (k >> b) & m, lo = k & m;
  return c == 0 ? k : c == 1 ? code_of(0, hi, lo, mid, b) : code_of(0, mid, hi, lo, b);
}

template <bool SAME_LINE>
__device__ __forceinline__ LinkPt link_point(int r, int n, int bits, int code, const int32_t* __restrict__ ord,
                                             const uint32_t* keys, const int2* __restrict__ rank12) {
  LinkPt q{-1, -1, 0u};
  if (r < 0 || r >= n) return q;
  const int2 id = link_id(r, n, code, ord, rank12);
  if (id.x < 0) return q;
  q.k = id.x;
  q.r2 = id.y;
  q.c = SAME_LINE ? c1_from_code(code, keys[r], bits) : keys[r];
  return q;
}

__device__ __forceinline__ LinkPt shfl_pt(LinkPt p, int delta, bool up) {
  LinkPt q;
  q.k = up ? __shfl_up_sync(0xffffffffu, p.k, delta) : __shfl_down_sync(0xffffffffu, p.k, delta);
  q.r2 = up ? __shfl_up_sync(0xffffffffu, p.r2, delta) : __shfl_down_sync(0xffffffffu, p.r2, delta);
  q.c = up ? __shfl_up_sync(0xffffffffu, p.c, delta) : __shfl_down_sync(0xffffffffu, p.c, delta);
  return q;
}

constexpr int kLinkThreads = 256;
constexpr int kLinkPerLane = 4;

// whether two points lie on one scan line of `code` (equal in its two major coordinates)
__device__ __forceinline__ bool same_scan_line(int code, uint32_t a, uint32_t c, int b) {
  int ax, ay, az, cx, cy, cz;
  decode_c1(a, b, ax, ay, az);
  decode_c1(c, b, cx, cy, cz);
  if (code == 0) return az == cz && ay == cy;
  if (code == 1) return ax == cx && az == cz;
  return ay == cy && ax == cx;
}

// Under the same-line variant (same_line) a pair is linked along a code only on
// one scan line of it (k_c1_line_flags then records the missing C1 links).
template <bool SAME_LINE>
__device__ __forceinline__ void link_body(const LinkArgs& la, int bx, int gx, int code) {
  const int n = la.n, bits = la.bits, cap = la.cap;
  const int32_t* __restrict__ ord23 = la.ord23;
  const uint32_t* __restrict__ keys_c2 = la.keys_c2;
  const uint32_t* __restrict__ keys_c3 = la.keys_c3;
  const int2* __restrict__ rank12 = la.rank12;
  const uint32_t* __restrict__ pk = la.pk;
  int4* __restrict__ c4 = la.c4;
  DevScalars* __restrict__ sc = la.sc;
  __shared__ unsigned long long s_red[8];
  const int lane = threadIdx.x & 31;
  const int32_t* ord = code == 0 ? nullptr : ord23 + size_t(code - 1) * size_t(cap);
  const uint32_t* keys = code == 0 ? pk : (code == 1 ? keys_c2 : keys_c3);
  const bool vec = ((reinterpret_cast<uintptr_t>(ord) | reinterpret_cast<uintptr_t>(keys)) & 15u) == 0;
  unsigned long long edges = 0;
  float dist_f = 0.f;  // this thread's few edge lengths; converted to fixed point once
  constexpr int kSpan = 32 * kLinkPerLane;
  const int warps = gx * (kLinkThreads / 32);
  // whole warps step together so the shuffles see every lane
  for (int base = (bx * (kLinkThreads / 32) + (threadIdx.x >> 5)) * kSpan; base < n; base += warps * kSpan) {
    const int r0 = base + kLinkPerLane * lane;
    int kk[kLinkPerLane];
    uint32_t cc[kLinkPerLane];
    if (vec && r0 + kLinkPerLane <= n) {
      const uint4 kv = *reinterpret_cast<const uint4*>(keys + r0);
      cc[0] = kv.x;
      cc[1] = kv.y;
      cc[2] = kv.z;
      cc[3] = kv.w;
      if (code == 0) {
#pragma unroll
        for (int i = 0; i < kLinkPerLane; ++i) kk[i] = r0 + i;
      } else {
        const int4 ov = *reinterpret_cast<const int4*>(ord + r0);
        kk[0] = ov.x;
        kk[1] = ov.y;
        kk[2] = ov.z;
        kk[3] = ov.w;
      }
    } else {
#pragma unroll
      for (int i = 0; i < kLinkPerLane; ++i) {
        const int r = r0 + i;
        kk[i] = -1;
        cc[i] = 0u;
        if (r < n) {
          kk[i] = code == 0 ? r : ord[r];
          cc[i] = keys[r];
        }
      }
    }
    if (code == 0 && la.colors.rgb && r0 < n) colors_quad(la.colors, r0, n);
    LinkPt p[kLinkPerLane];
#pragma unroll
    for (int i = 0; i < kLinkPerLane; ++i) {
      // (code 0: the position is the sorted id; else kk holds the input index)
      const bool in = in_range(kk[i], n);
      p[i].k = kk[i];
      p[i].r2 = -1;
      if (code == 1) p[i].k = in ? rank12[kk[i]].x : -1;
      if (code == 2) {
        const int2 q = in ? rank12[kk[i]] : make_int2(-1, -1);
        p[i].k = q.x;
        p[i].r2 = q.y;
      }
      p[i].c = SAME_LINE ? c1_from_code(code, cc[i], bits) : cc[i];
    }
#pragma unroll
    for (int i = 0; i < kLinkPerLane; ++i)
      if (!in_range(p[i].k, n)) p[i].k = -1;
    LinkPt before = shfl_pt(p[kLinkPerLane - 1], 1, true);
    LinkPt after = shfl_pt(p[0], 1, false);
    if (lane == 0) before = link_point<SAME_LINE>(r0 - 1, n, bits, code, ord, keys, rank12);
    if (lane == 31) after = link_point<SAME_LINE>(r0 + kLinkPerLane, n, bits, code, ord, keys, rank12);
#pragma unroll
    for (int i = 0; i < kLinkPerLane; ++i) {
      const LinkPt me = p[i];
      const LinkPt prev = i == 0 ? before : p[i - 1];
      const LinkPt next = i == kLinkPerLane - 1 ? after : p[i + 1];
      if (me.k < 0) continue;
      constexpr bool sl = SAME_LINE;
      const bool next_ok = next.k >= 0 && (!sl || same_scan_line(code, me.c, next.c, bits));
      const bool prev_ok = prev.k >= 0 && (!sl || same_scan_line(code, me.c, prev.c, bits));
      // the edge to the next position: counted once, unless an earlier code links the pair
      // (C1: adjacent sorted ids; C2: adjacent C2 positions; each on one line under the variant)
      bool dup_next = true;
      if (next_ok) {
        dup_next = code > 0 && abs(me.k - next.k) == 1 && (!sl || same_scan_line(0, me.c, next.c, bits));
        if (code == 2) dup_next |= abs(me.r2 - next.r2) == 1 && (!sl || same_scan_line(1, me.c, next.c, bits));
        if (!dup_next) {
          edges += 1;
          dist_f += sqrtf(float(sq_dist_c1(me.c, next.c, bits)));
        }
      }
      if (code == 0) continue;
      bool dup_prev = true;
      if (prev_ok) {
        dup_prev = abs(me.k - prev.k) == 1 && (!sl || same_scan_line(0, me.c, prev.c, bits));
        if (code == 2) dup_prev |= abs(me.r2 - prev.r2) == 1 && (!sl || same_scan_line(1, me.c, prev.c, bits));
      }
      int2* slot = reinterpret_cast<int2*>(c4 + me.k) + (code - 1);
      *slot = make_int2(dup_prev ? -1 : prev.k, dup_next ? -1 : next.k);
    }
  }
  unsigned long long dist = (unsigned long long)__float2ull_rn(dist_f * float(1u << kDistShift));
  edges = block_sum_u64<kLinkThreads>(edges, s_red);
  dist = block_sum_u64<kLinkThreads>(dist, s_red);
  if (threadIdx.x == 0) {
    if (edges) atomicAdd(&sc->n_edges, edges);
    if (dist) atomicAdd(&sc->dist_fx, dist);
  }
}

// Resident blocks per SM, and so registers a thread (48): with 6 (40) the loop spilled,
// and 16 segmented frames of 20k-100k points took 39 us, now 33; with 4 35, with 8 41.
constexpr int kLinkPerSm = 5;

template <bool SAME_LINE>
__global__ void __launch_bounds__(kLinkThreads, kLinkPerSm) k_link(LinkArgs a) {
  pdl_wait();
  link_body<SAME_LINE>(a, blockIdx.x, gridDim.x, blockIdx.y);
}

// segmented: frame f's blocks are three runs of equal length, one per code
template <bool SAME_LINE>
__global__ void __launch_bounds__(kLinkThreads, kLinkPerSm) k_link_seg(const __grid_constant__ Seg<LinkArgs> s) {
  pdl_wait();
  const int f = seg_frame(s, blockIdx.x);
  const int local = blockIdx.x - s.start[f], gx = (s.start[f + 1] - s.start[f]) / 3;
  link_body<SAME_LINE>(s.a[f], local % gx, gx, local / gx);
}

// Same-line variant: the missing links of every sorted point to its C1
// neighbours k - 1, k + 1 (not on its C1 scan line) go into the high bits of
// its packed code, where every kernel that takes k +- 1 as neighbours looks.
// (A neighbour's word may already carry its own bits when read: the
// coordinates are decoded through masks, so that does not matter.)
// `colors`: the colours that were taken into C1 order with their codes (rgb null: none).
__device__ __forceinline__ void c1_line_flags_body(int n, int bits, uint32_t* pk, const ColorArgs& colors, int bid,
                                                   int nblk) {
  for (int k = bid * blockDim.x + threadIdx.x; k < n; k += nblk * blockDim.x) {
    const uint32_t c = pk[k] & kCoordMask;
    const bool prev_ok = k > 0 && same_scan_line(0, c, pk[k - 1], bits);
    const bool next_ok = k + 1 < n && same_scan_line(0, c, pk[k + 1], bits);
    const uint32_t w = c | (prev_ok ? 0u : kNoPrevLink) | (next_ok ? 0u : kNoNextLink);
    pk[k] = w;
    if (colors.rgb && colors.pk) {
      if (colors.dtype != 0) reinterpret_cast<uint32_t*>(colors.yf + k)[3] = w;
      else if (colors.pc) colors.pc[k].x = w;
    }
  }
}

__global__ void __launch_bounds__(256) k_c1_line_flags(int n, int bits, uint32_t* pk, ColorArgs colors) {
  pdl_wait();
  c1_line_flags_body(n, bits, pk, colors, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(256) k_c1_line_flags_seg(const __grid_constant__ Seg<LinkArgs> s) {
  pdl_wait();
  const int f = seg_frame(s, blockIdx.x);
  c1_line_flags_body(s.a[f].n, s.a[f].bits, s.a[f].pk, s.a[f].colors, blockIdx.x - s.start[f], s.start[f + 1] - s.start[f]);
}

// Windows w > 1 (Section 2.2 with w points linked on each side): one thread
// per (code l, position r) fills the slots of the point at r for code l, the
// points d = 1..w positions before and after it: C2/C3 d = 1 into c4, every
// code's d >= 2 into cx (C1 d = 1 stays implicit: k - 1, k + 1).  A pair that
// an earlier code links (C1: sorted ids at most w apart; C2: C2 positions at
// most w apart; each on one scan line under the same-line variant) is left
// out of the later code's slots, so the union graph is a set.  The decision
// is a function of the pair and the code, so both ends reach the same one.
// Each undirected edge is counted (and its length summed) once, from the
// earlier position.  The points of a tile and of the w positions on either side of
// it are looked up once, into shared memory (each is read 2 w + 1 times; gathered
// for each pair anew, 400,000 points took 35 us with w = 2, now 27).
__global__ void __launch_bounds__(256) k_link_wide(ColorArgs colors, int n, int bits, int cap, int window,
                                                  int same_line,
                                                  const int32_t* __restrict__ ord23,
                                                  const uint32_t* __restrict__ keys_c2,
                                                  const uint32_t* __restrict__ keys_c3,
                                                  const int2* __restrict__ rank12, const uint32_t* __restrict__ pk,
                                                  int4* __restrict__ c4, int32_t* __restrict__ cx, int cx_stride,
                                                  DevScalars* __restrict__ sc) {
  pdl_wait();
  __shared__ unsigned long long s_red[8];
  const int code = blockIdx.y;
  const int32_t* ord = code == 0 ? nullptr : ord23 + size_t(code - 1) * size_t(cap);
  const uint32_t* keys = code == 0 ? pk : (code == 1 ? keys_c2 : keys_c3);
  const bool sl = same_line != 0;
  unsigned long long edges = 0;
  float dist_f = 0.f;
  constexpr int kTile = 256, kSpan = kTile + 2 * kMaxWindow;
  __shared__ int s_k[kSpan], s_r2[kSpan];
  __shared__ uint32_t s_c[kSpan];
  for (int base = blockIdx.x * kTile; base < n; base += gridDim.x * kTile) {
    __syncthreads();  // the tile before has been read
    for (int e = threadIdx.x; e < kTile + 2 * window; e += kTile) {
      const int rr = base - window + e;
      int2 id = make_int2(-1, -1);
      uint32_t c = 0u;
      if (rr >= 0 && rr < n) {
        id = link_id(rr, n, code, ord, rank12);
        c = c1_from_code(code, keys[rr] & kCoordMask, bits);
      }
      s_k[e] = id.x;
      s_r2[e] = id.y;
      s_c[e] = c;
    }
    if (code == 0 && colors.rgb && threadIdx.x < kTile / 4 && base + 4 * int(threadIdx.x) < n)
      colors_quad(colors, base + 4 * int(threadIdx.x), n);  // (four points a thread)
    __syncthreads();
    const int at = threadIdx.x + window;  // this thread's position, base + threadIdx.x
    const int k = s_k[at];
    if (k < 0) continue;  // (also behind the last position; the barriers come before, for every thread)
    const uint32_t c = s_c[at];
    const int r2 = s_r2[at];
    for (int d = 1; d <= window; ++d) {
      int slot[2];
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        slot[side] = -1;
        const int oe = side ? at + d : at - d;
        const int o = s_k[oe];
        if (o < 0) continue;
        const uint32_t oc = s_c[oe];
        if (sl && !same_scan_line(code, c, oc, bits)) continue;
        bool dup = false;
        if (code >= 1) dup = abs(k - o) <= window && (!sl || same_scan_line(0, c, oc, bits));
        if (code == 2 && !dup) {
          const int o2 = s_r2[oe];
          dup = abs(r2 - o2) <= window && (!sl || same_scan_line(1, c, oc, bits));
        }
        if (dup) continue;
        slot[side] = o;
        if (side) {
          edges += 1;
          dist_f += sqrtf(float(sq_dist_c1(c, oc, bits)));
        }
      }
      if (d == 1) {
        if (code > 0) reinterpret_cast<int2*>(c4 + k)[code - 1] = make_int2(slot[0], slot[1]);
      } else {
        const int s0 = 6 * (d - 2) + 2 * code;
        cx[size_t(s0) * size_t(cx_stride) + k] = slot[0];
        cx[size_t(s0 + 1) * size_t(cx_stride) + k] = slot[1];
      }
    }
  }
  unsigned long long dist = (unsigned long long)__float2ull_rn(dist_f * float(1u << kDistShift));
  edges = block_sum_u64<256>(edges, s_red);
  dist = block_sum_u64<256>(dist, s_red);
  if (threadIdx.x == 0) {
    if (edges) atomicAdd(&sc->n_edges, edges);
    if (dist) atomicAdd(&sc->dist_fx, dist);
  }
}

// Each sorted point's mean edge length (its neighbours from every slot), for
// the node and pair readings of sigma_g: written to node_sig (if set), and its
// fixed-point sum over the points that have edges, with their count, added to
// the build scalars.
__global__ void __launch_bounds__(256) k_node_sigma(int n, int bits, GraphBufs gb, DevScalars* __restrict__ sc) {
  pdl_wait();
  __shared__ unsigned long long s_red[8];
  unsigned long long sum = 0, cnt = 0;
  const int slots = 6 + gb.nx;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const uint32_t pkw = gb.pk[k];
    const int4 s4 = gb.c4[k];
    float len = 0.f;
    int deg = 0;
    for (int j = 0; j < slots; ++j) {
      const int o = neighbour_of(j, k, n, pkw, s4, gb.cx, gb.cx_stride);
      if (o < 0) continue;
      len += sqrtf(float(sq_dist_c1(pkw, gb.pk[o], bits)));
      deg += 1;
    }
    const float mean = deg ? len / float(deg) : 0.f;
    if (gb.node_sig) gb.node_sig[k] = mean;
    if (deg) {
      sum += __float2ull_rn(mean * float(1u << kDistShift));
      cnt += 1;
    }
  }
  sum = block_sum_u64<256>(sum, s_red);
  cnt = block_sum_u64<256>(cnt, s_red);
  if (threadIdx.x == 0) {
    if (sum) atomicAdd(&sc->node_fx, sum);
    if (cnt) atomicAdd(&sc->node_cnt, cnt);
  }
}

// The three orders in input indices.
__global__ void __launch_bounds__(256) k_orders_export(int n, int cap, const int32_t* __restrict__ perm1,
                                                       const int32_t* __restrict__ ord23, int32_t* __restrict__ out) {
  pdl_wait();
  const int stride = gridDim.x * blockDim.x;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += stride) {
    out[r] = perm1[r];
    out[size_t(n) + r] = ord23[r];
    out[2 * size_t(n) + r] = ord23[size_t(cap) + r];
  }
}

}  // namespace

namespace {
// blocks of one frame's launch of each kernel (the same in both paths)
// one 4096-point tile a block, up to two resident blocks per SM
int coord_hist_blocks(int n, int num_sms) {
  return n <= 0 ? 0 : std::max(1, std::min((n + kSortTile - 1) / kSortTile, 2 * num_sms));
}
int link_gx(int n, int num_sms) {
  // up to two blocks per SM for each of the three codes.  Five of those six are resident at a
  // time (kLinkPerSm), so above 311,000 points a sixth of the blocks starts as others end.
  // The number of blocks decides which edge lengths a thread adds in float32, so it is the
  // same in both paths.
  return std::max(1, std::min((n + kLinkThreads * kLinkPerLane - 1) / (kLinkThreads * kLinkPerLane), num_sms * 2));
}
int line_flag_blocks(int n, int num_sms) { return n <= 0 ? 0 : std::min((n + 255) / 256, num_sms * 8); }

// blocks of the row scatter: enough to fill the GPU twice while a tile keeps at least 1024
// points (each block pays for a scan of the rows and one global atomic a row)
int scatter_blocks(int n, int fill) {
  return n <= 0 ? 0 : std::max(std::min(fill, (n + 1023) / 1024), (n + kSortTile - 1) / kSortTile);
}
// output positions a block of the bucket sort owns: large windows share its fixed costs (scans,
// barriers, the rows' starts) over more points (300k points: 14.9 us at 4096, 16.7 at 2048; 217k:
// 13.3 at 2048, 15.1 at 1024), small frames keep enough blocks to spread over the SMs (20k: 6.7 us
// at 1024, 7.2 at 256)
int sort_window(int n) { return n >= (1 << 17) ? kWindowMax : n >= (1 << 15) ? kWindowMax / 2 : kWindowMax / 4; }
int sort_items(int n) { return n <= 0 ? 0 : (n + sort_window(n) - 1) / sort_window(n); }

template <int THREADS>
cudaError_t scatter_attr() {
  // the shared-memory limit is a per-device function attribute: set it once per device
  static std::atomic<unsigned long long> configured{0};
  return once_per_device(configured, [] {
    cudaError_t e = cudaFuncSetAttribute(k_bucket_scatter<THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(kScatterSmem));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_bucket_scatter_seg<THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               int(kScatterSmem));
    return e;
  });
}

cudaError_t sort_attr() {
  static std::atomic<unsigned long long> configured{0};  // the shared-memory limit is set once per device
  return once_per_device(configured, [] {
    cudaError_t e = cudaFuncSetAttribute(k_bucket_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kBucketSmem));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_bucket_sort_seg, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kBucketSmem));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_direct_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kBucketSmem));
    return e;
  });
}

template <typename A, typename K>
cudaError_t launch_seg(K kernel, const A* args, const int* blocks, int count, int threads, size_t smem,
                       cudaStream_t stream) {
  if (count < 1 || count > kSegMax) return cudaErrorInvalidValue;
  Seg<A> sg;
  for (int f = 0; f < count; ++f) sg.a[f] = args[f];
  const int grid = seg_layout(sg, blocks, count);
  if (grid == 0) return cudaSuccess;
  return launch_kernel(kernel, dim3(grid), dim3(threads), smem, stream, false, sg);
}

}  // namespace

HistArgs hist_args(const int32_t* xyz, int n, int bits, DevScalars* sc) { return HistArgs{xyz, n, bits, sc}; }

LinkArgs link_args(int n, int bits, int cap, const GraphBufs& gb, const SortBufs& sb, DevScalars* sc,
                   const ColorArgs& colors) {
  return LinkArgs{n, bits, cap, gb.ord23, sb.keys_c2, sb.keys_c3, gb.rank12, gb.pk, gb.c4, sc, colors};
}

BucketArgs bucket_args(const int32_t* xyz, int n, int bits, int cap, const SortBufs& sb, const GraphBufs& gb,
                       DevScalars* sc, int fill) {
  BucketArgs a{};
  a.xyz = xyz;
  a.n = n;
  a.bits = bits;
  const int blocks = scatter_blocks(n, fill);
  a.tile = blocks > 0 ? (n + blocks - 1) / blocks : 0;
  a.window = sort_window(n);
  for (int c = 0; c < 3; ++c) {
    a.row_pts[c] = sb.row_pts[c];
    a.row_tmp[c] = sb.row_tmp[c];
  }
  a.lines = sb.lines;
  a.line_slots = sb.line_slots;
  a.keys_out[0] = gb.pk;
  a.keys_out[1] = sb.keys_c2;
  a.keys_out[2] = sb.keys_c3;
  a.order_out[0] = gb.perm1;
  a.order_out[1] = gb.ord23;
  a.order_out[2] = gb.ord23 + size_t(cap);
  a.rank12 = reinterpret_cast<int32_t*>(gb.rank12);
  a.sc = sc;
  return a;
}

cudaError_t launch_coord_hist(const int32_t* xyz, int n, int bits, DevScalars* sc, int num_sms, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  // one block a tile, two per SM: every tile of a 1M-point frame in one wave
  return launch_kernel(k_coord_hist, dim3(coord_hist_blocks(n, num_sms)), dim3(1024), 0, stream, false,
                       hist_args(xyz, n, bits, sc));
}

cudaError_t launch_bucket_scatter(const BucketArgs& a, cudaStream_t stream) {
  if (a.n <= 0) return cudaSuccess;
  const cudaError_t e = scatter_attr<kScatterThreads>();
  if (e != cudaSuccess) return e;
  return launch_kernel(k_bucket_scatter<kScatterThreads>, dim3((a.n + a.tile - 1) / a.tile), dim3(kScatterThreads),
                       kScatterSmem, stream, false, a);
}

cudaError_t launch_bucket_sort(const BucketArgs& a, cudaStream_t stream) {
  if (a.n <= 0) return cudaSuccess;
  const cudaError_t e = sort_attr();
  if (e != cudaSuccess) return e;
  return launch_kernel(k_bucket_sort, dim3(sort_items(a.n), 3), dim3(kBucketThreads), kBucketSmem, stream, false, a);
}

cudaError_t launch_direct_sort(const BucketArgs& a, const ZeroArgs& z, cudaStream_t stream) {
  if (a.n <= 0 || a.n > kDirectMax) return cudaErrorInvalidValue;
  const cudaError_t e = sort_attr();
  if (e != cudaSuccess) return e;
  const int zero = std::max(1, int(std::min<size_t>((z.words + kBucketThreads - 1) / kBucketThreads, 64)));
  return launch_kernel(k_direct_sort, dim3(3 + zero), dim3(kBucketThreads), kBucketSmem, stream, false, a, z);
}

cudaError_t launch_link(int n, int bits, int cap, bool same_line, const GraphBufs& gb, const SortBufs& sb,
                        DevScalars* sc, const ColorArgs& colors, int num_sms, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int gx = link_gx(n, num_sms);
  const LinkArgs la = link_args(n, bits, cap, gb, sb, sc, colors);
  if (!same_line) return launch_kernel(k_link<false>, dim3(gx, 3), dim3(kLinkThreads), 0, stream, false, la);
  const cudaError_t e = launch_kernel(k_link<true>, dim3(gx, 3), dim3(kLinkThreads), 0, stream, false, la);
  if (e != cudaSuccess) return e;
  return launch_kernel(k_c1_line_flags, dim3(line_flag_blocks(n, num_sms)), dim3(256), 0, stream, false, n, bits,
                       gb.pk, colors);
}

// ---- segmented (one launch over the frames of a batch)

cudaError_t launch_coord_hist_seg(const HistArgs* a, int count, int num_sms, cudaStream_t stream) {
  int blocks[kSegMax];
  for (int f = 0; f < count && f < kSegMax; ++f) blocks[f] = coord_hist_blocks(a[f].n, num_sms);
  return launch_seg(k_coord_hist_seg, a, blocks, count, 1024, 0, stream);
}

cudaError_t launch_bucket_scatter_seg(const BucketArgs* a, int count, int scatter_threads, cudaStream_t stream) {
  int tiles[kSegMax];
  for (int f = 0; f < count && f < kSegMax; ++f) tiles[f] = a[f].n > 0 ? (a[f].n + a[f].tile - 1) / a[f].tile : 0;
  cudaError_t e;
  switch (scatter_threads) {
    case 256:
      e = scatter_attr<256>();
      return e != cudaSuccess ? e : launch_seg(k_bucket_scatter_seg<256>, a, tiles, count, 256, kScatterSmem, stream);
    case 1024:
      e = scatter_attr<1024>();
      return e != cudaSuccess ? e : launch_seg(k_bucket_scatter_seg<1024>, a, tiles, count, 1024, kScatterSmem, stream);
    default:
      e = scatter_attr<512>();
      return e != cudaSuccess ? e : launch_seg(k_bucket_scatter_seg<512>, a, tiles, count, 512, kScatterSmem, stream);
  }
}

cudaError_t launch_bucket_sort_seg(const BucketArgs* a, int count, cudaStream_t stream) {
  const cudaError_t e = sort_attr();
  if (e != cudaSuccess) return e;
  int blocks[kSegMax];
  for (int f = 0; f < count && f < kSegMax; ++f) blocks[f] = 3 * sort_items(a[f].n);
  return launch_seg(k_bucket_sort_seg, a, blocks, count, kBucketThreads, kBucketSmem, stream);
}

cudaError_t launch_link_seg(const LinkArgs* a, int count, bool same_line, int num_sms, cudaStream_t stream) {
  int blocks[kSegMax], flags[kSegMax];
  for (int f = 0; f < count && f < kSegMax; ++f) {
    blocks[f] = a[f].n > 0 ? 3 * link_gx(a[f].n, num_sms) : 0;
    flags[f] = line_flag_blocks(a[f].n, num_sms);
  }
  if (!same_line) return launch_seg(k_link_seg<false>, a, blocks, count, kLinkThreads, 0, stream);
  const cudaError_t e = launch_seg(k_link_seg<true>, a, blocks, count, kLinkThreads, 0, stream);
  if (e != cudaSuccess) return e;
  return launch_seg(k_c1_line_flags_seg, a, flags, count, 256, 0, stream);
}

cudaError_t launch_link_wide(int n, int bits, int cap, int window, bool same_line, const GraphBufs& gb,
                             const SortBufs& sb, DevScalars* sc, const ColorArgs& colors, int num_sms,
                             cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  if (window < 2 || window > kMaxWindow || gb.nx != extra_slots(window) || !gb.cx) return cudaErrorInvalidValue;
  const int gx = std::max(1, std::min((n + 255) / 256, num_sms * 4));
  const cudaError_t e = launch_kernel(k_link_wide, dim3(gx, 3), dim3(256), 0, stream, false, colors, n, bits, cap, window,
                                      same_line ? 1 : 0, gb.ord23, sb.keys_c2, sb.keys_c3, gb.rank12, gb.pk, gb.c4,
                                      gb.cx, gb.cx_stride, sc);
  if (e != cudaSuccess || !same_line) return e;
  return launch_kernel(k_c1_line_flags, dim3(std::min((n + 255) / 256, num_sms * 8)), dim3(256), 0, stream, false, n,
                       bits, gb.pk, colors);
}

cudaError_t launch_node_sigma(int n, int bits, const GraphBufs& gb, DevScalars* sc, int num_sms, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int grid = std::max(1, std::min((n + 255) / 256, num_sms * 8));
  return launch_kernel(k_node_sigma, dim3(grid), dim3(256), 0, stream, false, n, bits, gb, sc);
}

cudaError_t launch_orders_export(int n, int cap, const GraphBufs& gb, int32_t* out, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const int grid = std::max(1, std::min((n + 255) / 256, 152 * 16));
  return launch_kernel(k_orders_export, dim3(grid), dim3(256), 0, stream, false, n, cap, gb.perm1, gb.ord23, out);
}

// ---------------------------------------------------------------- shared launch pieces

bool pdl_enabled() {
  static const bool on = std::getenv("FGBD_PDL") != nullptr;
  return on;
}

namespace {
__global__ void __launch_bounds__(256) k_zero_words(uint32_t* __restrict__ p, size_t words) {
  pdl_wait();
  for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < words; i += size_t(gridDim.x) * blockDim.x)
    p[i] = 0u;
}

__global__ void __launch_bounds__(256) k_zero_words_seg(const __grid_constant__ Seg<ZeroArgs> s) {
  pdl_wait();
  const int f = seg_frame(s, blockIdx.x);
  const size_t b = size_t(blockIdx.x - s.start[f]), nb = size_t(s.start[f + 1] - s.start[f]);
  for (size_t i = b * blockDim.x + threadIdx.x; i < s.a[f].words; i += nb * blockDim.x) s.a[f].p[i] = 0u;
}
}  // namespace

cudaError_t launch_zero_words_seg(const ZeroArgs* a, int count, cudaStream_t stream) {
  int blocks[kSegMax];
  for (int f = 0; f < count && f < kSegMax; ++f) blocks[f] = int(std::min<size_t>((a[f].words + 255) / 256, 64));
  return launch_seg(k_zero_words_seg, a, blocks, count, 256, 0, stream);
}

cudaError_t launch_zero_words(uint32_t* p, size_t words, cudaStream_t stream) {
  if (words == 0) return cudaSuccess;
  const int grid = int(std::min<size_t>((words + 255) / 256, 64));
  return launch_kernel(k_zero_words, dim3(grid), dim3(256), 0, stream, false, p, words);
}

}  // namespace fgbd
