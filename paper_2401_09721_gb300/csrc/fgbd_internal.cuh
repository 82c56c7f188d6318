// Internal declarations shared by the FGBD CUDA translation units.
//
// Index spaces.  The caller's points are in "input order".  Internally every
// per-point array is kept in "sorted order": the order of the first scan-line
// code C1 = 2^{2b} z + 2^b y + x (Section 2.2, Eq. 1).  In that order the two
// code-1 neighbours of point k are simply k-1 and k+1, and the packed C1 code
// of point k doubles as its coordinates.  Neighbours along C2 and C3
// (Eq. 2-3) are stored explicitly, four slots per point, with -1 marking an
// empty slot (the end of a scan order, or a pair already linked by an earlier
// code, so that the union graph of Section 2.2 is a set).  With a window
// w > 1 the points d = 2..w positions away along each code are stored in
// 6 (w - 1) further slots per point (GraphBufs::cx).
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace fgbd {

constexpr int kMaxBits = 10;                       // three b-bit coordinates fit a 32-bit code
constexpr int kMaxRadix = 1 << kMaxBits;           // values of one coordinate (b bits)
constexpr int kSortTile = 4096;                    // points a block of the histogram / row scatter holds at most
constexpr int kK = 6;                              // neighbours per point at window 1
constexpr int kD = 3 * (kK + 1);                   // patch dimension (Section 2.3)
constexpr int kMaxWindow = 3;                      // windows 1..3: K = 6w neighbours per point
constexpr int kDMax = 3 * (6 * kMaxWindow + 1);    // largest patch dimension (57)
constexpr int kQCap = 256;                         // largest q_max accepted
constexpr int kSqShift = 8;                        // fixed point of squared colours (2^-8)
constexpr int kDistShift = 20;                     // fixed point of edge lengths
constexpr int kNeThreads = 256;
constexpr int kNeGroup = 32;                       // float colours: moment blocks whose sums their last block adds up
constexpr int kNeGroups = 32;                      // at most kNeGroup * kNeGroups moment blocks
constexpr int kFilterThreads = 512;
// Filter steps taken while sigma_est is computed: kSpecSure of them whatever that
// takes, and in contexts of up to kSpecSmall points as many as fit beside the eigen
// step (28 us), up to kSpecMax.  A step of 20,000 points takes 3 us there, and a grid
// barrier and as much again in the selection: with powers of 5 and 6 frames of 3,000
// and 20,000 points take 70 and 68 us, 84 and 81 with three stored steps.  One of
// 100,000 takes 4 us and the frames of that size stop earlier: 106 us, 104 with three.
constexpr int kSpecSure = 3;
constexpr int kSpecMax = 8;
constexpr int kSpecSmall = 1 << 16;
constexpr int spec_rows(int64_t cap) { return cap <= kSpecSmall ? kSpecMax : kSpecSure; }
constexpr uint32_t kCoordMask = 0x3FFFFFFFu;       // low 30 bits: packed C1 code
// The two high bits of a sorted point's packed code (pk, and x.w of an iterate)
// mark a missing link to its C1 neighbour k - 1 / k + 1: set by the link step
// only under the same-line variant, zero otherwise.
constexpr uint32_t kNoPrevLink = 1u << 30;
constexpr uint32_t kNoNextLink = 1u << 31;
constexpr uint32_t kKeepBit = 0x80000000u;         // FSLR keep flag beside the code

// latched device error bits
enum : uint32_t {
  kFlagRange = 1u,    // a coordinate outside [0, 2^b)
  kFlagTimeout = 2u,  // a bounded device-side wait gave up
};

// Device-resident scalars of one context.  Regions are zeroed separately by
// the call that fills them (see the offsets used in api.cu).
struct DevScalars {
  // ---- graph build region
  unsigned long long n_edges;   // distinct undirected edges E
  unsigned long long dist_fx;   // sum of edge lengths, fixed point 2^-kDistShift
  alignas(16) uint32_t chist[3][kMaxRadix];  // histograms of x, y and z
  unsigned long long node_fx;   // node-mean reading: sum over points of their mean edge length (fixed point)
  unsigned long long node_cnt;  // and the points that have edges
  float cexp;                   // the Eq. 4 exponent scale log2(e) / sigma_g^2 of this graph, once cexp_ready
  uint32_t cexp_ready;          // set by the first moments launch on this graph
  uint32_t row_used[3][kMaxRadix];  // row scatter: places of every x, y and z row handed out so far
  uint32_t row_ext[3][2];           // per coordinate: 2^b - 1 minus its smallest value, and its largest
  // codes with rows above kRowSplit points (k_bucket_sort): blocks take turns by tickets, and
  // how many of those rows have their counters cleared, and of their points are counted and placed
  uint32_t sort_ticket[3], rows_cleared[3], lines_counted[3], lines_placed[3];
  uint32_t build_end_;
  // ---- noise estimate region
  unsigned long long n_patches;
  long long s1[kD];             // sum of (a - 128)
  long long s2[kD * kD];        // sum of (a - 128)(a - 128)^T (upper triangle filled)
  uint32_t ne_groups[kNeGroups];  // float colours: blocks of each group that have written their moments
  uint32_t spec_barrier;        // grid barrier of the speculative filter steps
  int32_t spec_done;            // filter steps stored by the noise-estimate kernel
  uint32_t sigma_ready;         // set (release) once sigma_est of this estimate is written
  uint32_t sigma_near;          // set when it is a few microseconds away: no further speculative step
  uint32_t spec_go[kSpecMax + 1];  // after stored step t: 1 to take another before selecting
  float fslr_thr[4];            // the FSLR threshold of this sigma_est as the selection uses it (once fslr_ready)
  uint32_t fslr_ready;          // set by the eigen step with sigma_est
  uint32_t ne_end_;
  // ---- results of the noise estimate
  double eig[kDMax];            // descending (the first D = 3 (6w + 1) are used)
  double tau;
  double sigma_est;
  int32_t m;
  int32_t ne_valid;
  // ---- selection region
  unsigned long long ysq_keep;  // fixed point 2^-kSqShift
  unsigned long long ysq_all;
  unsigned long long n_keep;
  unsigned long long sumsq[kQCap + 1];
  long long spec_keep[kSpecMax + 1];  // over the kept points: sum of x_q^2 (fixed point), stored steps q = 1..
  long long spec_all[kSpecMax + 1];   // the same over every point
  uint32_t barrier;
  uint32_t barrier_rest;        // of the launch that takes the search up again
  int32_t resume_t;             // the step after which a segmented launch left the search to it (0: it did not)
  uint32_t sel_end_;
  // ---- results of the selection
  double J[kQCap + 1];
  int32_t kept_buf;             // where x_q is: 0 / 1 the iterate buffers, 2 + q - 1 a stored step, -1 the input,
                                // kKeptBest the copy of the global reading's best iterate
  int32_t q_sel;
  int32_t n_J;
  int32_t sel_valid;
  // ---- latched errors (never zeroed by a call; cleared when read)
  uint32_t status;
  uint32_t row_start[3][kMaxRadix + 1];  // row scatter: first place of every x, y and z row, then n (not zeroed)
  // ---- settings (set at context creation)
  unsigned long long wait_limit_ns;  // any device-side wait gives up after this long
  uint32_t sigma_mode;               // sigma_g of Eq. 4: kSigmaEdge, kSigmaNode or kSigmaPair
  uint32_t pooled_patch;             // 1: patches of D = 7 pooled over the colour channels (Section 2.3)
  double fslr_factor;                // the FSLR threshold factor (2 in Section 2.4)
};

// Readings of sigma_g (Section 2.2): the mean length over the edges (the
// method as read here), the mean over the points of each point's mean edge
// length, or a bandwidth per point (w_ij = exp(-d_ij^2 / (sigma_i sigma_j))).
enum : uint32_t { kSigmaEdge = 0u, kSigmaNode = 1u, kSigmaPair = 2u };

// the regions are zeroed as 32-bit words
static_assert(offsetof(DevScalars, n_edges) % 4 == 0 && offsetof(DevScalars, build_end_) % 4 == 0 &&
                  offsetof(DevScalars, n_patches) % 4 == 0 && offsetof(DevScalars, ne_end_) % 4 == 0 &&
                  offsetof(DevScalars, ysq_keep) % 4 == 0 && offsetof(DevScalars, sel_end_) % 4 == 0,
              "DevScalars regions must be whole 32-bit words");
static_assert(offsetof(DevScalars, n_edges) < offsetof(DevScalars, build_end_) &&
                  offsetof(DevScalars, build_end_) < offsetof(DevScalars, n_patches) &&
                  offsetof(DevScalars, ne_end_) < offsetof(DevScalars, ysq_keep),
              "the build, noise and selection regions are zeroed as one range by fgbd_run");

// Sort scratch for one build.  row_pts and row_tmp may share memory with arrays
// that are only used after the graph is built (the stored filter steps).
struct SortBufs {
  uint2* row_pts[3];     // per code [cap]: (input index, code) of every point, row by row
  uint2* row_tmp[3];     // per code [cap]: the points of split rows line by line; the long-item sort's scratch
  uint32_t* lines;       // [3][line_slots][2][kMaxRadix]: the line counters of split rows (kRowSplit)
  int line_slots;
  uint32_t* keys_c2;     // [cap] the C2 codes along C2
  uint32_t* keys_c3;     // [cap] the C3 codes along C3
};

// Graph in sorted order.
struct GraphBufs {
  int32_t* perm1;    // [cap] input index of each sorted (C1-order) point
  int2* rank12;      // [cap] of each input point: its sorted id (x) and its position in the C2 order (y)
  uint32_t* pk;      // [cap] packed C1 code of each sorted point (its coordinates)
  int32_t* ord23;    // [2][cap] input indices along C2, then along C3
  int4* c4;          // [cap] C2 prev, C2 next, C3 prev, C3 next (sorted ids, -1 empty)
  // windows w > 1: [6 (w - 1)][cap stride] the points d = 2..w positions away;
  // slot 6 (d - 2) + 2 l + s holds code l's point d before (s = 0) / after (s = 1)
  // the point (sorted ids, -1 empty or linked by an earlier code)
  int32_t* cx;
  int nx;            // 6 (w - 1)
  int cx_stride;     // row stride of cx, a multiple of 64
  float* node_sig;   // [cap] each sorted point's mean edge length (the node and pair readings of sigma_g), or null
};

// number of further neighbour slots at window w
__host__ __device__ constexpr int extra_slots(int w) { return 6 * (w - 1); }

// A row of more points than this is put line by line before it is sorted (k_bucket_sort).
// Its counters, [2][kMaxRadix] points a line (counted, then placed), are those number
// (first place) / (kRowSplit + 1) of its code: two such rows start further apart than that.
constexpr int kRowSplit = 32768;
constexpr int line_slots(int64_t cap) { return int(cap / (kRowSplit + 1)) + 1; }
constexpr size_t line_words(int64_t cap) { return size_t(3) * size_t(line_slots(cap)) * 2 * kMaxRadix; }

// The row scatter and the bucket sort of one frame (codes 0 C1, 1 C2, 2 C3).
struct BucketArgs {
  int n;
  int bits;
  int tile;                // points per block of the scatter
  int window;              // output positions per block of the sort
  const int32_t* xyz;
  uint2* row_pts[3];       // SortBufs
  uint2* row_tmp[3];
  uint32_t* lines;
  int line_slots;
  uint32_t* keys_out[3];   // code c of the points along code c
  int32_t* order_out[3];   // the input indices along each code
  int32_t* rank12;         // GraphBufs::rank12, as [n][2]
  DevScalars* sc;
};

// ---------------------------------------------------------------- segmented launches
// A batch of frames runs each stage as one launch: the per-frame arguments of
// up to kSegMax frames travel in the kernel's parameter space, and frame f
// owns the blocks [start[f], start[f + 1]) of a one-dimensional grid.  A
// block finds its frame, then runs the same body as the one-frame kernel with
// its block index and block count inside the frame, so a frame's results do
// not depend on the batch it is in.
constexpr int kSegMax = 16;

template <typename A>
struct Seg {
  A a[kSegMax];
  int start[kSegMax + 1];
  int count;
};

// the frame that owns block b (frames with no blocks are skipped)
template <typename A>
__device__ __forceinline__ int seg_frame(const Seg<A>& s, int b) {
  int f = 0;
  while (f + 1 < s.count && s.start[f + 1] <= b) ++f;
  return f;
}

// fill s.start from per-frame block counts; returns the grid size
template <typename A>
inline int seg_layout(Seg<A>& s, const int* blocks, int count) {
  s.count = count;
  int t = 0;
  for (int f = 0; f < count; ++f) {
    s.start[f] = t;
    t += blocks[f];
  }
  s.start[count] = t;
  return t;
}

// Arguments of the kernels that the one-frame path passes one by one.
struct HistArgs {
  const int32_t* xyz;
  int n;
  int bits;
  struct DevScalars* sc;
};
// The caller's colours (input order) and where they go in C1 order.
struct ColorArgs {
  const void* rgb;       // null: none
  int dtype;             // 0: uint8 into y8, else float32 into yf
  const int32_t* perm1;
  uint32_t* y8;
  float4* yf;
  uint2* pc;             // window 1, uint8: also (packed code, colour) of every sorted point, which the moments
                         // launch gathers as one word pair; null: not written
  const uint32_t* pk;    // window 1: the packed codes of the sorted points, the fourth word of yf (null: zero)
};
struct LinkArgs {
  int n;
  int bits;
  int cap;
  const int32_t* ord23;
  const uint32_t* keys_c2;
  const uint32_t* keys_c3;
  const int2* rank12;
  uint32_t* pk;
  int4* c4;
  struct DevScalars* sc;
  ColorArgs colors;
};
struct MomentArgs {
  int n;
  int bits;
  const uint2* pc;   // uint8: (packed code, colour) per sorted point
  const float4* yf;  // float: (R, G, B, packed code) per sorted point
  float4* x0;        // uint8: x_0 of the filter steps, (R, G, B, packed code), written here
  const int4* c4;
  float* spread;
  double* f64_partials;
  int sorted_patches;
  int per_sm;        // blocks of the launch on an SM, where they fill the GPU (else 1)
  int shares;        // float: shares of the points, one or two a block (ne_moment_shares)
  struct DevScalars* sc;
};
struct ZeroArgs {
  uint32_t* p;
  size_t words;
};

// How a batch runs, chosen by the batch tuner (api.cu): frames per segmented
// launch (0: every frame on a stream of its own, its own kernels), threads of
// the row scatter (a tile of up to 4096 points a block), threads of the filter blocks
// and filter blocks per SM of the cooperative selection.
struct BatchShape {
  int seg_frames = kSegMax;
  int scatter_threads = 512;
  int filter_threads = 512;
  int filter_per_sm = 2;
};

// ---------------------------------------------------------------- launchers
struct FilterArgs;
// Every launcher enqueues on `stream` and returns the launch error.

// the coordinate histograms (and the range check)
cudaError_t launch_coord_hist(const int32_t* xyz, int n, int bits, DevScalars* sc, int num_sms, cudaStream_t stream);
// `cap`: distance between the C2 and the C3 half of gb.ord23; `fill`: blocks of the row scatter that
// fill the GPU (or this frame's share of it)
BucketArgs bucket_args(const int32_t* xyz, int n, int bits, int cap, const SortBufs& sb, const GraphBufs& gb,
                       DevScalars* sc, int fill);
constexpr int scatter_fill(int num_sms) { return 2 * num_sms; }  // two resident blocks per SM
cudaError_t launch_bucket_scatter(const BucketArgs& a, cudaStream_t stream);
cudaError_t launch_bucket_sort(const BucketArgs& a, cudaStream_t stream);
// a frame of up to kDirectMax points in one launch, from the coordinates; it also zeroes z
constexpr int kDirectMax = 8192;
cudaError_t launch_direct_sort(const BucketArgs& a, const ZeroArgs& z, cudaStream_t stream);
cudaError_t launch_orders_export(int n, int cap, const GraphBufs& gb, int32_t* out, cudaStream_t stream);
// segmented launches: one launch for frames 0..count-1 (count <= kSegMax).  The histogram,
// the sort, the link and the float moments give each frame the blocks its one-frame launch
// would have; the row scatter and the uint8 moments its share of the blocks that fill the
// GPU, which changes no result (the order inside a row is the sort's, the moments are
// exact integers)
HistArgs hist_args(const int32_t* xyz, int n, int bits, DevScalars* sc);
LinkArgs link_args(int n, int bits, int cap, const GraphBufs& gb, const SortBufs& sb, DevScalars* sc,
                   const ColorArgs& colors);
cudaError_t launch_zero_words_seg(const ZeroArgs* a, int count, cudaStream_t stream);
cudaError_t launch_coord_hist_seg(const HistArgs* a, int count, int num_sms, cudaStream_t stream);
// (scatter_threads: 256, 512 or 1024 per tile)
cudaError_t launch_bucket_scatter_seg(const BucketArgs* a, int count, int scatter_threads, cudaStream_t stream);
cudaError_t launch_bucket_sort_seg(const BucketArgs* a, int count, cudaStream_t stream);
cudaError_t launch_link_seg(const LinkArgs* a, int count, bool same_line, int num_sms, cudaStream_t stream);
cudaError_t launch_link(int n, int bits, int cap, bool same_line, const GraphBufs& gb, const SortBufs& sb,
                        DevScalars* sc, const ColorArgs& colors, int num_sms, cudaStream_t stream);
// each sorted point's mean edge length into gb.node_sig (if set) and, for the
// node reading of sigma_g, their sum and count into the build scalars
cudaError_t launch_node_sigma(int n, int bits, const GraphBufs& gb, DevScalars* sc, int num_sms, cudaStream_t stream);
// windows w > 1: every link of the window (C2/C3 d = 1 into c4, d >= 2 into cx)
// and the edge sums; then k_c1_line_flags under the same-line variant
cudaError_t launch_link_wide(int n, int bits, int cap, int window, bool same_line, const GraphBufs& gb,
                             const SortBufs& sb, DevScalars* sc, const ColorArgs& colors, int num_sms,
                             cudaStream_t stream);

cudaError_t launch_gather_colors(const ColorArgs& a, int n, cudaStream_t stream);
cudaError_t launch_ne_moments(const MomentArgs& a, int dtype, int num_sms, cudaStream_t stream);
// spec: if not null (and spec->spec_depth > 0), the same launch also takes the
// first spec_depth filter steps on the other SMs (one block per SM)
cudaError_t launch_ne_finalize(int dtype, const double* f64_partials, int nblocks,
                               DevScalars* sc, double* sigma_out, const FilterArgs* spec, int num_sms,
                               cudaStream_t stream);
int ne_moment_shares(int n, int num_sms);
int ne_moment_blocks(int n, int num_sms, int dtype);
// testing: div_newton and CUDA's division of n operand pairs
cudaError_t launch_debug_div(const double* a, const double* b, double* q_newton, double* q_div, int64_t n,
                             cudaStream_t stream);
// segmented: frames 0..count-1 (count <= kSegMax; one colour dtype for the moments)
cudaError_t launch_ne_moments_seg(const MomentArgs* a, int count, int dtype, int num_sms, cudaStream_t stream);
// the estimate launch over frames: one eigen block per frame, the other SMs
// shared out for the speculative steps (spec[f].spec_depth of them)
cudaError_t launch_ne_finalize_seg(const FilterArgs* spec, const double* const* f64_partials, const int* nblocks,
                                   int count, int num_sms, cudaStream_t stream);

// Noise estimate at windows w > 1 (patch dimension D = 3 (6w + 1)): per-block
// moment partials, their reduction, the one-block float32 eigenvectors, and float64
// Rayleigh quotients with the tail rule.
struct WideNe {
  double* part;   // [blocks][D*D + D + 1] per-block moments (int64 bit patterns for uint8 colours)
  double* tot;    // [D*D + D + 1] the totals: sum a a^T (upper triangle), sum a, patch count
  double* S;      // [D][D] the covariance
  float* V;       // [D][D] its eigenvector estimates (columns), then their D float32 eigenvalues
  double* lam;    // [D] Rayleigh quotients
  uint32_t* done; // blocks of the Rayleigh launch finished (reset by the last)
  int blocks;     // moment blocks (the rows of part)
};
int ne_wide_blocks(int n, int num_sms);
size_t ne_wide_part_entries(int window);  // D*D + D + 1
// stage 0 the moments (nothing at n = 0), 1 their reduction, 2 the eigenvector block, 3 the tail rule
cudaError_t launch_ne_wide(int stage, int n, int bits, int window, int dtype, const GraphBufs& gb,
                           const uint32_t* y8, const float4* yf, float* spread, const WideNe& w, DevScalars* sc,
                           double* sigma_out, int num_sms, cudaStream_t stream);

struct FilterArgs {
  int n;
  int bits;
  int dtype;             // colours held in y8 (0) or yf (1)
  int mode;              // 0: select q (Eq. 6), 1: fixed q
  int q_fixed;           // mode 1
  const int32_t* q_src;  // mode 1: if set, q is read here on the device (and q_sel is left as it is)
  int q_max;             // mode 0
  int step_cap;          // segmented launch: the step after which it leaves the search (0: none)
  double fslr_factor;
  int all_points;        // Eq. 6 over every point (the limited region is off)
  const double* sigma_src;  // sigma_est to use (device)
  const uint32_t* y8;
  const float4* yf;
  const float* spread;
  const uint32_t* pk;
  const int4* c4;
  const int2* rank12;    // (x: the sorted id of each input point)
  float4* xbuf0;
  float4* xbuf1;
  void* out;             // input-order output or nullptr
  int out_dtype;
  DevScalars* sc;
  // select mode: the first spec_depth steps were stored before sigma_est was known
  int spec_depth;          // 0: none
  const float4* x0;        // x_0 (r, g, b, packed code): float colours themselves, or as the moments launch wrote
                           // it into xbuf0; null: from y8, pk
  float4* spec_x;          // [spec_rows(cap)][cap]: x_1 .. x_S
  int32_t* spec_z;         // [spec_rows(cap)][cap]: per point sum_c x_q^2, fixed point
  int cap;                 // row stride of spec_x / spec_z, a multiple of 64
  int fuse;                // noise-estimate launch: select and filter too, once sigma_est is known
  uint8_t* keep8;          // select mode: the FSLR keep flag of every sorted point
  // windows w > 1: the further neighbour slots (GraphBufs::cx), nx = 6 (w - 1)
  const int32_t* cx;
  int nx;
  int cx_stride;
  // the pair reading of sigma_g: each sorted point's mean edge length (null otherwise)
  const float* node_sig;
  // the global reading of the q search: argmin of J over 0..q_max; the best
  // iterate beyond the stored steps is copied to xbest
  int q_global;
  float4* xbest;
  // window 1: the Eq. 4 weights of each sorted point's six slots, normalised by
  // their sum (slots C1 prev, C1 next, C2 prev, C2 next in w4; C3 prev, next in
  // w2), written by step 1 and read by every later step of the same graph
  float4* w4;
  float2* w2;
  int32_t* dmin;           // windows w > 1: each point's smallest squared distance, left by step 1
};
constexpr int kKeptBest = 64;  // kept_buf value of the iterate copied to xbest
cudaError_t launch_filter(const FilterArgs& a, int grid, cudaStream_t stream);
int filter_grid(int n, int num_sms, int nx = 0);
cudaError_t launch_output(const FilterArgs& a, cudaStream_t stream);  // the kept iterate, in input order
// the cooperative selection/filter over frames (window 1): filter_per_sm blocks
// of `threads` (256 or 512) per SM, shared out in proportion to the frames' points
cudaError_t launch_filter_seg(const FilterArgs* a, int count, int threads, int filter_per_sm, int num_sms,
                              cudaStream_t stream);
int filter_seg_max_per_sm(int threads);  // resident blocks per SM of that kernel
// the searches that it left (FilterArgs::step_cap), one frame after another with the whole GPU
cudaError_t launch_filter_rest_seg(const FilterArgs* a, int count, int num_sms, cudaStream_t stream);

// Differentiable filter: rows of R = D^-1 W for given alpha, sigma, and their transpose
struct DiffBufs {  // one value a neighbour slot: C1 (i - 1, i + 1) in the float2, C2/C3 in the float4
  float2* r2;   // [n] R_ij; -1: no neighbour
  float4* r4;   // [n]
  int4* rec;    // [n] packed code, smallest squared distance, 1 / sum of weights (bits)
  float2* rt2;  // [n] R_ji: weight of i in the row of its neighbour (backward)
  float4* rt4;  // [n]
  float2* g2;   // [n] R_ij (d_ij^2 - sum_k R_ik d_ik^2) (backward)
  float4* g4;   // [n]
};
int diff_grid(int n, int num_sms);
cudaError_t launch_diff_rows(int n, int bits, double sigma, const float* rgb, const GraphBufs& gb,
                             const DevScalars* sc, const DiffBufs& db, float4* x, int num_sms, cudaStream_t stream);
cudaError_t launch_diff_rows_t(int n, int bits, double sigma, const float* grad, const GraphBufs& gb,
                               const DevScalars* sc, const DiffBufs& db, float4* u, int num_sms, cudaStream_t stream);
cudaError_t launch_diff_scatter(int n, const float4* x, const int32_t* perm1, float* out, int num_sms,
                                cudaStream_t stream);
// out / grad_in: the result in input order (the last step), or null
cudaError_t launch_diff_step(int n, float alpha, const GraphBufs& gb, const DiffBufs& db, const float4* src,
                             float4* dst, float* out, int num_sms, cudaStream_t stream);
cudaError_t launch_diff_back_step(int n, float alpha, bool first, const GraphBufs& gb, const DiffBufs& db,
                                  const float4* x, const float4* u, float4* u_out, float* grad_in, double2* partial,
                                  int num_sms, cudaStream_t stream);
cudaError_t launch_diff_reduce(int count, float alpha, double sigma, const DevScalars* sc, const double2* partial,
                               double* grad, cudaStream_t stream);

// CSR export in input order
// row_ptr[0..n]; block_tmp: a word per 1024 rows and one more, which the fill reads
cudaError_t launch_csr_row_ptr(int n, const GraphBufs& gb, int64_t* row_ptr, int64_t* block_tmp,
                               const DevScalars* sc, cudaStream_t stream);
cudaError_t launch_csr_fill(int n, int bits, const GraphBufs& gb, const int64_t* row_ptr, const int64_t* block_tmp,
                            int32_t* col, float* w, int64_t col_capacity, const DevScalars* sc, cudaStream_t stream);
cudaError_t launch_spread_export(int n, const int2* rank12, const float* spread, const uint8_t* keep8,
                                 float* spread_out, uint8_t* keep_out, cudaStream_t stream);

// ---------------------------------------------------------------- device helpers

__host__ __device__ inline uint32_t code_of(int which, uint32_t x, uint32_t y, uint32_t z, int b) {
  // Eq. 1-3 with the three b-bit fields packed high to low
  switch (which) {
    case 0: return (z << (2 * b)) | (y << b) | x;
    case 1: return (x << (2 * b)) | (z << b) | y;
    default: return (y << (2 * b)) | (x << b) | z;
  }
}

// an index read from device memory is used only if it lies in [0, n)
__device__ __forceinline__ bool in_range(int v, int n) { return unsigned(v) < unsigned(n); }

// Colour of input point i (R, G, B in the low three bytes) out of n: from the one
// or two aligned words that hold its bytes, where the array starts on a word
// and the second word lies inside it (three byte loads a point fill the load
// queue: 10.8 us at 1M points).
__device__ __forceinline__ uint32_t load_rgb8(const uint8_t* __restrict__ rgb, uint32_t i, uint32_t n, bool words) {
  const size_t at = 3 * size_t(i);
  if (words && i + 2 < n) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(rgb) + (at >> 2);
    const uint32_t off = uint32_t(at) & 3u;
    const uint32_t lo = __ldg(w), hi = off > 1u ? __ldg(w + 1) : 0u;
    return __funnelshift_r(lo, hi, 8u * off) & 0xffffffu;
  }
  return uint32_t(__ldg(rgb + at)) | (uint32_t(__ldg(rgb + at + 1)) << 8) | (uint32_t(__ldg(rgb + at + 2)) << 16);
}
__device__ __forceinline__ float4 load_rgbf(const float* __restrict__ rgb, uint32_t i) {
  const size_t at = 3 * size_t(i);
  return make_float4(__ldg(rgb + at), __ldg(rgb + at + 1), __ldg(rgb + at + 2), 0.f);
}

// The colours of the sorted points k0 .. k0 + 3 (k0 a multiple of 4) below n into
// C1 order: their input indices read as one int4 and the loads issued together.
__device__ __forceinline__ void colors_quad(const ColorArgs& a, int k0, int n) {
  int pi[4];
  if (k0 + 4 <= n) {
    const int4 v = *reinterpret_cast<const int4*>(a.perm1 + k0);
    pi[0] = v.x;
    pi[1] = v.y;
    pi[2] = v.z;
    pi[3] = v.w;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) pi[i] = k0 + i < n ? a.perm1[k0 + i] : -1;
  }
  uint32_t p[4] = {0u, 0u, 0u, 0u};
  if (a.pk) {
    if (k0 + 4 <= n) {
      const uint4 v = *reinterpret_cast<const uint4*>(a.pk + k0);
      p[0] = v.x;
      p[1] = v.y;
      p[2] = v.z;
      p[3] = v.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (k0 + i < n) p[i] = a.pk[k0 + i];
    }
  }
  if (a.dtype == 0) {
    const uint8_t* rgb = static_cast<const uint8_t*>(a.rgb);
    const bool words = (reinterpret_cast<uintptr_t>(rgb) & 3u) == 0;
    uint32_t c[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) c[i] = in_range(pi[i], n) ? load_rgb8(rgb, uint32_t(pi[i]), uint32_t(n), words) : 0u;
    if (k0 + 4 <= n) {
      *reinterpret_cast<uint4*>(a.y8 + k0) = make_uint4(c[0], c[1], c[2], c[3]);
      if (a.pc) {
        uint4* pc = reinterpret_cast<uint4*>(a.pc + k0);
        pc[0] = make_uint4(p[0], c[0], p[1], c[1]);
        pc[1] = make_uint4(p[2], c[2], p[3], c[3]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (k0 + i < n) {
          a.y8[k0 + i] = c[i];
          if (a.pc) a.pc[k0 + i] = make_uint2(p[i], c[i]);
        }
    }
  } else {
    const float* rgb = static_cast<const float*>(a.rgb);
    float4 c[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      c[i] = in_range(pi[i], n) ? load_rgbf(rgb, uint32_t(pi[i])) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (k0 + i < n) a.yf[k0 + i] = make_float4(c[i].x, c[i].y, c[i].z, __uint_as_float(p[i]));
  }
}

__device__ __forceinline__ void decode_c1(uint32_t c, int b, int& x, int& y, int& z) {
  const uint32_t m = (1u << b) - 1u;
  x = int(c & m);
  y = int((c >> b) & m);
  z = int((c >> (2 * b)) & m);
}

// whether sorted point k is linked to k - 1 / k + 1 (C1 neighbours), from its packed-code word
__device__ __forceinline__ bool c1_prev_linked(uint32_t pkw, int k) { return k > 0 && !(pkw & kNoPrevLink); }
__device__ __forceinline__ bool c1_next_linked(uint32_t pkw, int k, int n) { return k + 1 < n && !(pkw & kNoNextLink); }

// Neighbour j (0 .. 5 + nx) of sorted point k in link order: 0 / 1 the C1
// points k - 1 / k + 1 (pkw: k's packed-code word with the missing-link
// bits), 2..5 the c4 slots s, then the further slots of a window w > 1.
// Returns its sorted id, or -1 for an empty slot.
__device__ __forceinline__ int neighbour_of(int j, int k, int n, uint32_t pkw, int4 s, const int32_t* __restrict__ cx,
                                            int cx_stride) {
  int v;
  switch (j) {
    case 0: return c1_prev_linked(pkw, k) ? k - 1 : -1;
    case 1: return c1_next_linked(pkw, k, n) ? k + 1 : -1;
    case 2: v = s.x; break;
    case 3: v = s.y; break;
    case 4: v = s.z; break;
    case 5: v = s.w; break;
    default: v = cx[size_t(j - 6) * size_t(cx_stride) + k]; break;
  }
  return in_range(v, n) ? v : -1;
}

__device__ __forceinline__ int sq_dist_c1(uint32_t a, uint32_t c, int b) {
  int ax, ay, az, cx, cy, cz;
  decode_c1(a, b, ax, ay, az);
  decode_c1(c, b, cx, cy, cz);
  const int dx = cx - ax, dy = cy - ay, dz = cz - az;
  return dx * dx + dy * dy + dz * dz;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s for any device-side wait

__device__ __forceinline__ uint32_t ld_volatile(const uint32_t* p) {
  return *reinterpret_cast<const volatile uint32_t*>(p);
}
__device__ __forceinline__ void st_volatile(uint32_t* p, uint32_t v) {
  *reinterpret_cast<volatile uint32_t*>(p) = v;
}

// round(v^2 * 2^kSqShift) as a 32-bit integer: exact for integer colours,
// within 2^-9 otherwise; colours on the 0..255 scale (|v| < 2896) fit.
// A 32-bit conversion keeps the per-point work off the float64 pipe.
__device__ __forceinline__ int sq_fixed(float v) { return __float2int_rn(v * v * float(1 << kSqShift)); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// block-wide sum of a 64-bit counter, result valid in thread 0
template <int THREADS>
__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v,
                                                            unsigned long long* smem) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) smem[warp] = v;
  __syncthreads();
  unsigned long long t = 0;
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) t += smem[w];
  }
  __syncthreads();
  return t;
}

// sigma_g (Section 2.2) from the build sums: the mean edge length, or under
// the node reading the mean of the points' mean edge lengths
__device__ __forceinline__ double sigma_g_of(const DevScalars* sc) {
  if (sc->sigma_mode == kSigmaNode) {
    const unsigned long long c = sc->node_cnt;
    return c ? double(sc->node_fx) * (1.0 / double(1ull << kDistShift)) / double(c) : 0.0;
  }
  const unsigned long long e = sc->n_edges;
  if (e == 0) return 0.0;
  return double(sc->dist_fx) * (1.0 / double(1ull << kDistShift)) / double(e);
}

// ---------------------------------------------------------------- launches
// Programmatic dependent launch (opt-in): with FGBD_PDL set in the
// environment, consecutive kernels are launched with programmatic stream
// serialization.  Every kernel starts with pdl_wait(), which then returns once
// the kernel it depends on has completed and its writes are visible; under an
// ordinary launch it returns at once.  Measured on the 1M-point frame it
// gained nothing (0.2635 vs 0.2632 ms), and letting the next kernel launch at
// the start of each kernel cost 12 us (waiting blocks held resources the
// multi-wave kernels needed), so ordinary launches are the default.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

bool pdl_enabled();  // true if the environment sets FGBD_PDL

// Launch `kernel` on `stream`: cooperative (all blocks resident, for the grid
// barriers) or with programmatic stream serialization.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                 bool cooperative, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attrs[1];
  cfg.attrs = attrs;
  cfg.numAttrs = 0;
  if (cooperative) {
    attrs[0].id = cudaLaunchAttributeCooperative;
    attrs[0].val.cooperative = 1;
    cfg.numAttrs = 1;
  } else if (pdl_enabled()) {
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 1;
  }
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Run `set` (a kernel attribute change, which is idempotent) once per device:
// `done` holds one bit per device index.  Safe from several host threads; two
// threads may both run `set` the first time, which changes nothing.
template <typename F>
inline cudaError_t once_per_device(std::atomic<unsigned long long>& done, F&& set) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = set();
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_acq_rel);
  return e;
}

// zero [p, p + words) on `stream` (a kernel, so it joins the programmatic chain)
cudaError_t launch_zero_words(uint32_t* p, size_t words, cudaStream_t stream);

}  // namespace fgbd
