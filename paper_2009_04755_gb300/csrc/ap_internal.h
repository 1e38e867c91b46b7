// ap_internal.h -- internal declarations of the all-pairs library.
//
// Storage kept by a handle, the launch wrappers of each kernel family and the
// host planners.  Nothing here is part of the C ABI (see allpairs.h).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <atomic>
#include <functional>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "allpairs.h"

namespace ap {

// ---------------------------------------------------------------------------
// status word written by bounded device waits (AP device error codes)
// ---------------------------------------------------------------------------
enum DeviceError : int32_t {
  DEV_OK = 0,
  DEV_TIMEOUT_FULL = 1,     // consumer gave up waiting for a stage to fill
  DEV_TIMEOUT_EMPTY = 2,    // producer gave up waiting for a stage to drain
  DEV_TIMEOUT_ACCUM = 3,    // epilogue gave up waiting for the accumulator
  DEV_TIMEOUT_STAGE = 4,    // a bulk copy of item data did not land
  DEV_TIMEOUT_SLOT = 5,     // a slot-ready flag was never raised
  DEV_TIMEOUT_UNIT = 6,     // a CTA pair's unit hand-out ring did not advance
};

// wall-clock budget of one device wait (nanoseconds, %globaltimer)
constexpr unsigned long long kWaitBudgetNs = 2000000000ull;   // 2 s

// ---------------------------------------------------------------------------
// packed upper-triangle index, p(i,j) = i*n - i(i+1)/2 + (j-i-1)
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ int64_t pair_index(int64_t i, int64_t j, int64_t n) {
  return i * n - (i * (i + 1)) / 2 + (j - i - 1);
}

// float -> double on the integer pipe: GB300 converts on its FP64 pipe, two
// values per clock and SM, which an epilogue of 32,768 sums a CTA feels
#ifdef __CUDACC__
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m != 0) return (double)x;   // subnormal, infinite, NaN
  const uint32_t hi = (u & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
  return __hiloint2double((int)hi, (int)(u << 29));
}
#endif

// ---------------------------------------------------------------------------
// point-cloud storage: items sorted by the planner, padded to a multiple of
// 4 points, held in pairs of points so that one packed FP32x2 operation takes
// two of them as they lie: pair q (points 2q, 2q + 1) is
//   2-D  {x0, x1, y0, y1} {s0, s1, l0, l1}
//   3-D  {x0, x1, y0, y1} {z0, z1, s0, s1}, and {l0, l1} in lw[]
// with s = s2k = -sigma^2 / (log2(e)/2) (negated) and l = log2(weight) (-inf
// for padding), so that
//   w_b * exp(-d^2 / (2 (sa^2 + sb^2))) = 2^(l_b + d^2 / (s_a + s_b)).
// ---------------------------------------------------------------------------
//
// In a boxed set, the points of an item of more than kCullPoints are stored
// in an order that keeps neighbours together (cloud_pack_kernel), and every 32
// of them have a box: {xmin, xmax, ymin, ymax} {zmin, zmax, largest |s2k|,
// largest log-weight}, so that a warp passes over 32 points at once where all
// its terms with them are 0 in FP32 (2^x below 2^-126).  Boxes of item i
// (storage position) start at cloud_box0(first group of i, i).
//
// What boxes save hangs on how far the Gaussians reach against the extent of
// the items; looking at them costs 2-6%.  A set is boxed from a mean of
// kBoxedMean points on (over points, so that large items count).  Times without
// boxes over those with them, clouds over [-1, 1]^dim with sigma 0.01-0.03 /
// 0.02-0.05:
//   points      2-D overlap    its adjoint    2-D GMM L2     3-D overlap
//   200-300     0.98 / 0.96    1.02 / 0.97    1.01 / 0.95    1.15 / 0.99
//   400-600     1.18 / 0.96    1.19 / 0.98    1.23 / 1.00    0.98 / 0.96
//   600-760     1.32 / 1.04    1.30 / 1.03    1.34 / 1.06    1.04 / 0.97
//   800-1200    1.52 / 1.16    1.50 / 1.14    1.54 / 1.18    1.15 / 1.00
//   2000-3000   2.06 / 1.33    2.06 / 1.32    2.13 / 1.37    1.80 / 1.10
// and 50-5000 lognormal (1240 over points) 1.31 / 1.08 in 2-D, 1.16 / 1.02 in
// 3-D; GMM L2 of 256 particles of 1000-2000 points 22.1 -> 12.1 ms.  Putting the
// points in order takes part of a set's creation (1000 lognormal 3-D clouds 2.0
// -> 2.3 ms).  Terms of one size then follow one another, which the sums allow for
// (kBlockwise, kTree).
// An item of up to kCullPoints fills a warp or little more: no part of it is far
// from the rest.
constexpr int64_t kCullPoints = 160;
constexpr double kBoxedMean = 800.0;
__host__ __device__ __forceinline__ int64_t cloud_box0(int64_t grp0, int64_t i) {
  return grp0 / 8 + i;                 // a box per 8 groups, and one to spare per item
}
// The a-side of the pair sums.  Four consecutive storage points (a group)
// belong to one item; a warp job holds R points per lane.  An item's groups
// split into fragments by its own size alone: runs of 8 R groups, each filling
// a warp, then pieces of up to 8 groups.  Pieces of a block's items share
// warps (four pieces of 8 groups at R = 4), so the lanes stay filled at any
// item size; one partial sum per fragment and partner (a row).
__host__ __device__ __forceinline__ int32_t cloud_rows(int64_t cnt, int32_t R) {
  const int64_t g = (cnt + 3) / 4, full = 8 * R;
  return (int32_t)(g / full + (g % full + 7) / 8);
}
// Lane descriptor: x = group of four storage points (-1: idle), y = row (10
// bits), lane's place in its fragment (5), lanes of the fragment - 1 (5), item
// of the block (5), points per lane 1 << re (2), first point of the group in
// units of them (2).
__host__ __device__ __forceinline__ int32_t pack_lane(int32_t row, int32_t t, int32_t len,
                                                      int32_t il, int32_t re, int32_t sub) {
  return row | t << 10 | (len - 1) << 15 | il << 20 | re << 25 | sub << 27;
}
// points per lane (as a power of two) of a job with `pieces` pieces of 8 groups
__host__ __device__ __forceinline__ int32_t job_re(int32_t pieces) {
  return pieces <= 1 ? 0 : pieces == 2 ? 1 : 2;
}
// lane `lane` of job k of a single item of G groups starting at group grp0
__host__ __device__ __forceinline__ int2 cloud_lane_desc(int32_t k, int32_t lane, int32_t grp0,
                                                         int32_t G, int32_t R, int32_t row0,
                                                         int32_t il) {
  const int32_t full = 8 * R, nfull = G / full;
  int2 d;
  if (k < nfull) {
    const int32_t lpg = 4 / R;
    d.x = grp0 + k * full + lane / lpg;
    d.y = pack_lane(row0 + k, lane, 32, il, R == 4 ? 2 : 1, lane % lpg);
    return d;
  }
  const int32_t rem = G - nfull * full, re = job_re((rem + 7) / 8), lpg = 4 >> re;
  const int32_t gl = lane / lpg, in = gl < rem, left = rem - (gl & ~7);
  d.x = in ? grp0 + nfull * full + gl : -1;
  d.y = pack_lane(in ? row0 + nfull + (gl >> 3) : 0, in ? (gl & 7) * lpg + lane % lpg : 0,
                  in ? (left < 8 ? left : 8) * lpg : 1, il, re, lane % lpg);
  return d;
}

// a tile plan of a cloud set (plan.cpp): blocks, their warp jobs, the tiles
struct CloudPlanHost {
  std::vector<int32_t> bstart;      // block b = storage items [bstart[b], bstart[b+1])
  std::vector<int32_t> bmeta;       // [blocks][8]: item begin, end, first group, groups,
                                    // first job (-1: one item, see cloud_lane_desc), jobs,
                                    // rows, 0; then the single items that tiles split at the
                                    // end of the list take as their J side
  std::vector<int32_t> desc;        // [jobs][32][2] lane descriptors
  std::vector<int32_t> items;       // per stored item {first group, points, original id,
                                    // first row in its block}
  std::vector<int32_t> tiles;       // block pairs (I <= J), indices into bmeta
  int32_t max_rows = 1, max_items = 1, max_pts = 4;
  bool largest_first = false;
};

struct CloudStore {
  int dim = 2;
  int64_t n = 0;
  std::vector<int64_t> h_size;      // points per item (original order)
  std::vector<int32_t> h_perm;      // storage position -> original item id
  std::vector<int64_t> h_poff;      // padded offsets in storage order [n+1]
  int64_t total_pts = 0;            // padded
  float4 *d_pts = nullptr;          // [total_pts]
  float *d_lw = nullptr;            // [total_pts] (3-D only)
  bool boxed = false;               // large items in an order of neighbours, with boxes
  float4 *d_boxes = nullptr;        // [total_pts / 32 + n + 1][2] (boxed sets only)
  int64_t *d_poff = nullptr;        // [n+1]
  int32_t *d_cnt = nullptr;         // [n] real points per stored item
  int32_t *d_perm = nullptr;        // [n] storage position -> original item id
  // tile plan (rebuilt when the tuned parameters change)
  int32_t block_items = 0, block_pts = 0, reg_r = 0;
  int32_t max_rows = 0, max_items = 0, max_pts = 0;   // of any block
  bool sorted = false;
  // pair lists: tiles are listed pairs of one-item blocks, outputs by list
  // position (set only on the temporary copy a list run launches with)
  bool list_mode = false;
  std::vector<int32_t> h_iperm;     // original item id -> storage position
  int32_t *d_bmeta_single = nullptr;    // [n][8]: block b = item b
  int32_t *d_list_tiles = nullptr;  // [list_cap][2] storage positions
  int64_t list_cap = 0;
  int32_t *d_bmeta = nullptr;       // as in CloudPlanHost
  int32_t *d_desc = nullptr;
  int32_t *d_items = nullptr;
  int32_t *d_tiles = nullptr;       // [n_tiles][2] block pairs (I <= J)
  int64_t n_tiles = 0;
  // launch shapes already looked up for this plan's buffers (shared with the
  // temporary copies a list run or the tuner launches with)
  struct Fit { const void *kern; size_t smem; int threads; int64_t slots; };
  std::shared_ptr<std::vector<Fit>> fits = std::make_shared<std::vector<Fit>>();
  // particle scores: re-scaled storage per score (index score - 1), built on
  // first use, and the GMM L2 self terms per original item
  float4 *d_pts_score[2] = {nullptr, nullptr};
  float *d_lw_score[2] = {nullptr, nullptr};
  double *d_self = nullptr;
};

// one macro pair (a <= b) of an out-of-core batch and the slots holding them
struct OocPair { int32_t a, b, slot_a, slot_b; };
// one step of the out-of-core schedule: loads (macro, slot), then a Gram batch
struct OocStep {
  std::vector<std::pair<int32_t, int32_t>> loads;
  std::vector<OocPair> pairs;
  int64_t unit0 = 0, n_units = 0, cover0 = 0, n_cover = 0;
};

// ---------------------------------------------------------------------------
// dense-vector storage
// ---------------------------------------------------------------------------
constexpr int64_t kOocMacroItems = 256;   // items per device / host cache slot

// the second-level (host) cache of decoded macros and its parse threads
// (hostcache.cu)
struct HostCacheRelease;
struct HostCache {
  struct Impl;
  int64_t n = 0, dim = 0, n_slots = 0;
  size_t slot_floats = 0;
  const uint8_t *const *blobs = nullptr;
  const uint64_t *blob_bytes = nullptr;
  int32_t codec = 0;
  float *pinned = nullptr;                 // [n_slots][256][dim]
  Impl *impl = nullptr;
  HostCacheRelease *release_args = nullptr;
  // counters (under the lock)
  int64_t hits = 0, misses = 0, parsed_rows = 0;
  bool bad_input = false;
  ~HostCache();
  ap_status init(int64_t n_items, int64_t dim, const uint8_t *const *blobs,
                 const uint64_t *bytes, int32_t codec, int64_t slots, int threads);
  void announce(const std::vector<int64_t> &macros);   // the run's requests, in order
  int acquire(int64_t macro);                           // a ready slot, held
  void release(int slot);
  const float *slot_ptr(int slot) const { return pinned + (size_t)slot * slot_floats; }
  void *release_arg(int slot);
  static void CUDART_CB release_cb(void *arg);          // cudaLaunchHostFunc target
  void worker();
  void pump();
};
int64_t xor_varint_encode(const float *x, int64_t dim, uint8_t *out, uint64_t cap);
bool xor_varint_decode(const uint8_t *in, uint64_t len, int64_t dim, float *x);

struct VecStore {
  int64_t n = 0, D = 0, ld = 0;
  int64_t Dp = 0;                   // padded row length (multiple of 64)
  uint32_t precisions = 0;
  double *d_mu = nullptr, *d_ss = nullptr, *d_rs = nullptr;   // FP64 per item (d_mu: the shift)
  double *d_delta_all = nullptr;    // mean - shift per item
  double *d_partc = nullptr;        // [n][kSplitParts] partial sums of c
  double *d_part = nullptr;         // [n][kSplitParts] partial sums of c^2
  int64_t n_rows_alloc = 0;         // rows rounded up to the row block
  __nv_bfloat16 *d_hi = nullptr, *d_lo = nullptr;              // [n][Dp]
  float *d_c32 = nullptr;                                      // [n][Dp]
  uint8_t *d_list = nullptr;        // pair lists' index arrays and partial sums
  size_t list_bytes = 0;
  float *d_stage = nullptr;         // raw rows staged from the host
  int64_t stage_rows = 0;
  // out-of-core mode: HBM slot cache of 256-item macros
  bool out_of_core = false;
  const float *h_src = nullptr;
  HostCache *host = nullptr;        // encoded items: decoded macros in pinned host slots
  uint64_t slot_cache_bytes = 0;
  int64_t n_macros = 0, n_slots = 0, group = 0, ring = 0;
  __nv_bfloat16 *d_pool_hi = nullptr, *d_pool_lo = nullptr;   // slot pool, blocked layout
  float *d_raw = nullptr;                                      // raw staging ring
  std::vector<cudaEvent_t> ev_raw_ready, ev_raw_free, ev_prepped;
  std::vector<int> ring_used;
  std::vector<OocStep> steps;
  int32_t *d_units = nullptr, *d_cover_units = nullptr;
  void *tmap_pool_hi = nullptr, *tmap_pool_lo = nullptr;
  int64_t ooc_loads = 0, ooc_uses = 0;
  // out-of-core, column-sliced schedule (AP_OOC_K_SLICED): every item's
  // chunk of slice_cols columns resident at once in one chunk buffer ([0])
  int32_t ooc_policy = 0;
  int64_t slice_cols = 0, n_slices = 0;
  __nv_bfloat16 *d_slice_hi[2] = {nullptr, nullptr}, *d_slice_lo[2] = {nullptr, nullptr};
  void *tmap_slice_hi[2] = {nullptr, nullptr}, *tmap_slice_lo[2] = {nullptr, nullptr};
  double *d_shift = nullptr, *d_part_c = nullptr, *d_delta = nullptr;
  int32_t *d_slice_units = nullptr; int64_t n_slice_units = 0;
  int32_t *d_slice_cover = nullptr; int64_t n_slice_cover = 0;   // one unit per tile
  cudaEvent_t ev_slice_ready[2] = {nullptr, nullptr}, ev_slice_done[2] = {nullptr, nullptr};
  // streamed load-and-run of a resident set: per macro column m, the split-K
  // units of the pairs (a <= m, m) on the resident blocked arrays
  // With stream_chunks > 1 the columns go in chunks of stream_chunk_cols,
  // and entry c * macros + m holds the units of macro column m over chunk c
  int32_t *d_stream_units = nullptr;
  std::vector<std::pair<int64_t, int64_t>> stream_cols;   // (first unit, units)
  int64_t stream_chunks = 0, stream_chunk_cols = 0;
  // tile plans
  int32_t *d_tiles_tc = nullptr;  int64_t n_tiles_tc = 0;
  // k_split > 0: the tiles run as split-K units in waves (panel_units)
  int32_t k_split = 0;
  int32_t *d_panel_units = nullptr; int64_t n_panel_units = 0;
  // mma_ctas = 2: the same schedule on CTA pairs (gram_tc2.cu): split-K units
  // in waves of tc2_pairs() macro pairs, and one unit per macro pair (whole
  // columns: k_split = 0 and coverage)
  int32_t mma_ctas = 2;
  int32_t *d_pair_units = nullptr; int64_t n_pair_units = 0;
  float *d_planes = nullptr;        // [n_planes][n (n - 1) / 2] partial Grams of d_pair_units;
  int64_t n_planes = 0;             // without them the units add into the output
  int32_t *d_pair_whole = nullptr; int64_t n_pair_whole = 0;
  std::vector<int32_t> h_tiles_tc;
  int32_t *d_tiles_f32 = nullptr; int64_t n_tiles_f32 = 0;
  void *tmap_hi = nullptr, *tmap_lo = nullptr;   // CUtensorMap (host copies)
  double *d_g64 = nullptr;          // FP64 partial sums of the tensor-core Gram
};

}  // namespace ap

namespace ap {
// task trace of a streamed pipeline (ap_set_trace): CUDA events at the start
// and end of every task, on the stream that runs it
struct TraceRec {
  int32_t stream = 0, stage = 0;
  int64_t index = 0;
  uint64_t bytes = 0;
  cudaEvent_t a = nullptr, b = nullptr;
};
struct Tracer {
  bool on = false;
  cudaEvent_t base = nullptr;
  std::vector<TraceRec> recs;
  void clear();
  // a new trace whose time zero is now on s (no-op when tracing is off)
  cudaError_t start(cudaStream_t s);
  // open a task on st; returns its record (-1 when off)
  int begin(int32_t stream, int32_t stage, int64_t index, uint64_t bytes, cudaStream_t st);
  void end(int rec, cudaStream_t st);
  ~Tracer() { clear(); }
};
// host-side range for tools that show NVTX (the enqueue of one stage)
struct NvtxRange {
  explicit NvtxRange(const char *name);
  ~NvtxRange();
};
}  // namespace ap

namespace ap {
// a captured launch sequence, replayed with cudaGraphLaunch
struct GraphKey {
  const void *a, *b, *c;           // buffers the sequence reads / writes
  float eta, fmin;
  int32_t n;
  bool operator==(const GraphKey &o) const {
    return a == o.a && b == o.b && c == o.c && eta == o.eta && fmin == o.fmin && n == o.n;
  }
};
struct GraphEntry {
  GraphKey key;
  uint64_t plan_version;
  cudaGraphExec_t exec;
};
}  // namespace ap

namespace ap {
// sparse vectors in CSR form over an index space of `dim` codes, cut into
// chunks of kSparseChunk codes; cptr[c][i] = first entry of row i with a
// code >= c * kSparseChunk, relative to the row's start (chunk-major, so the
// bounds of 32 consecutive rows in one chunk are one coalesced load)
constexpr int kSparseChunk = 4096;
constexpr int kSparseBlock = 128;    // items of a tile side
struct SparseStore {
  int64_t n = 0, dim = 0, nnz = 0, n_chunks = 0;
  int64_t *d_off = nullptr;
  int32_t *d_idx = nullptr;
  float *d_val = nullptr;
  int32_t *d_cptr = nullptr;        // [n_chunks + 1][n]
  double *d_rs = nullptr;           // 1 / sqrt(sum of squares), NaN for none
  int32_t *d_tiles = nullptr;       // block pairs (I <= J) of 128 items
  int64_t n_tiles = 0;
  int32_t *d_chunks = nullptr;      // [n_join + n_gather + n_dense]: chunks with
                                    // shared codes, by way
  int64_t n_join = 0, n_gather = 0, n_dense = 0;
  unsigned long long *d_heads = nullptr;   // unit queues of the three kernels
};
}  // namespace ap

struct ap_items {
  int32_t kind = 0;
  int device = 0;
  ap::CloudStore cl;
  ap::VecStore vec;
  ap::SparseStore sp;
  std::mutex list_mutex;            // over vec.d_list, until a list run has finished
  int32_t *d_status = nullptr;      // [0] device error code, [1..] scratch
  int32_t *d_queue = nullptr;       // device words, see kQueueTraits
  std::atomic<uint32_t> launches{0};     // launches given a queue head (take_queue)
  float *d_scratch = nullptr;       // generic scratch
  int64_t scratch_bytes = 0;
  ap_run_stats stats{};
  int32_t last_dev_error = 0;
  cudaStream_t copy_stream = nullptr;
  cudaStream_t prep_stream = nullptr;    // pre-processing of streamed macros (load-and-run)
  cudaStream_t graph_stream = nullptr;   // private stream the graphs are captured on
  cudaEvent_t ev_a = nullptr, ev_b = nullptr;
  uint64_t plan_version = 0;
  uint64_t wait_budget_ns = 0;          // 0 = the default budget
  int32_t debug = 0;                    // failure-path testing switches
  ap::Tracer trace;                     // task trace of the streamed pipelines
  std::vector<ap::GraphEntry> graphs;
};

namespace ap {

// ---------------------------------------------------------------------------
// words of a handle's d_queue block, and unit queues
// ---------------------------------------------------------------------------
// [0] unit-queue head of the launches that clear it themselves, [1] status word,
// [2] scratch, traits of a cloud set (some s2k or coordinate is outside the range
// in which two terms may share a reciprocal; some weight is not 1), two heads for
// captured launches, and a ring of heads.
constexpr int kQueueTraits = 3, kQueueCaptured = 4, kQueueRing = 64;
constexpr uint32_t kQueueHeads = 64;
constexpr int kQueueWords = kQueueRing + (int)kQueueHeads;
// The queue of one launch: `head` is 0 when the launch starts, and the launch
// clears `ahead`.  Launches take the heads of the ring in turn and clear the one
// half the ring on, so that a run costs no clearing of its own (a memset before
// a small set's one kernel takes 2 of 10 us), and whatever a head is left at (by a
// device wait that ran out, by runs that overlapped) is gone when it comes round.
struct UnitQueue {
  int32_t *words, *head, *ahead;
};
// the next head of the ring; where the stream is being captured, a head that a
// memset in front of the launch clears, since a replay finds it as it was left
cudaError_t take_queue(ap_items *it, cudaStream_t s, UnitQueue *q);
// a queue taken for a launch that does not take place: clears `ahead` in its
// stead and returns e
cudaError_t leave_queue(const UnitQueue &q, cudaStream_t s, cudaError_t e);

// ---------------------------------------------------------------------------
// host planners (plan.cpp)
// ---------------------------------------------------------------------------
// Upper-triangle block pairs (I <= J) of an nb x nb block grid in recursive
// quadrant order (split in four, recurse, skip empty quadrants).
void dc_block_pairs(int64_t nb, std::vector<int32_t> &out);
// Group storage-ordered items into blocks of at most max_items items and
// max_pts padded points (an item larger than max_pts forms its own block).
// Blocks of several items also respect max_rows partial rows (cloud_rows).
void make_blocks(const std::vector<int64_t> &poff, const std::vector<int64_t> &cnt,
                 int32_t max_items, int64_t max_pts, int32_t reg_r, int64_t max_rows,
                 std::vector<int32_t> &bstart);
// the whole tile plan: blocks, the packing of their items' pieces into warp
// jobs, and the tiles in the order they are popped, the last split_tail of
// them split into one tile per item of J
void make_cloud_plan(const std::vector<int64_t> &poff, const std::vector<int64_t> &cnt,
                     const std::vector<int32_t> &perm, int64_t split_tail, int32_t block_items,
                     int32_t block_pts, int32_t reg_r, CloudPlanHost &out);

// ---------------------------------------------------------------------------
// kernel launchers
// ---------------------------------------------------------------------------
// vectors (vec.cu)
// Blocked layout of the pre-processed copies: rows in blocks of 128 items,
// columns in blocks of kblk; one (row block, column block) tile is a
// contiguous 128 x kblk array, so every tile load is one contiguous run.
constexpr int kRowBlock = 128;
constexpr int kTcKBlock = 32;     // bf16 columns per block (64 bytes per row)
constexpr int kF32KBlock = 16;    // fp32 columns per block (64 bytes per row)
constexpr int kSplitParts = 16;   // FP64 partials of sum c^2 and sum c per row
__host__ __device__ __forceinline__ size_t blocked_offset(int64_t row, int64_t k, int64_t nkb,
                                                          int kblk) {
  return ((size_t)(row / kRowBlock) * nkb + (size_t)(k / kblk)) * ((size_t)kRowBlock * kblk) +
         (size_t)(row % kRowBlock) * kblk + (size_t)(k % kblk);
}
cudaError_t launch_vec_mean(const float *X, int64_t n, int64_t D, int64_t ld, double *mu,
                            cudaStream_t s);
// the load pipeline of vectors in one launch: per row a shift (the mean of
// evenly spread samples), then the centred split / FP32 copies and the FP64
// sums of c and c^2 in one pass, then delta = mean - shift, ss and rs; rows
// whose shift missed the mean by D delta^2 > ss / 64 are redone from the
// exact mean.  set_rows: the rows of the whole set (see prep_cluster).
cudaError_t launch_vec_prep(const float *X, int64_t row0, int64_t out_row0, int64_t n,
                            int64_t set_rows, int64_t D, int64_t ld, int64_t Dp,
                            __nv_bfloat16 *hi, __nv_bfloat16 *lo, float *c32, double *shift,
                            double *delta, double *ss, double *rs, cudaStream_t s);
// out[p] -= (D delta_i rs_i)(delta_j rs_j) over the packed triangle: the
// mean correction of pairs the Gram kernel already scaled by rs_i rs_j
cudaError_t launch_pair_correct(double *out, const double *rs, const double *delta, int64_t n,
                                int64_t D, cudaStream_t s);
// out[p] = (sum over r of planes[r][p] - D delta_i delta_j) rs_i rs_j; NaN for
// every pair where the status word is set
cudaError_t launch_pair_planes(double *out, const float *planes, int64_t k, const double *rs,
                               const double *delta, const int32_t *status, int64_t n, int64_t D,
                               cudaStream_t s);
// out[p] = (out[p] - D delta_i delta_j) rs_i rs_j over the packed triangle
cudaError_t launch_pair_finalize(double *out, const double *rs, const double *delta, int64_t n,
                                 int64_t D, cudaStream_t s);
// columns [col0, col0 + width) of rows row0.. (cols of them real, staged
// with leading dimension ld) centred on per-row shifts and split into blocked
// copies Dl columns wide; FP64 partials of c and c^2 accumulated per row
cudaError_t launch_vec_split_cols(const float *X, int64_t row0, int64_t n, int64_t cols,
                                  int64_t ld, int64_t width, int64_t col0, int64_t Dl,
                                  const double *shift, __nv_bfloat16 *hi, __nv_bfloat16 *lo,
                                  float *c32, double *part, double *part_c, int first_chunk,
                                  cudaStream_t s);
// per-row shifts of rows read where they are (X may be pinned host memory
// the device can address): the mean of 32 evenly spaced runs of 32 values
cudaError_t launch_vec_shift_runs(const float *X, int64_t n, int64_t D, int64_t ld,
                                  double *shift, cudaStream_t s);
// one column chunk [.., cols) of rows row0.., centred on per-row shifts (the
// rows' blocked copies hold cols_p >= cols columns); FP64 partials of
// sum c^2 and sum c are set (first_chunk) or accumulated per row
cudaError_t launch_vec_split_slice(const float *X, int64_t row0, int64_t n, int64_t cols,
                                   int64_t ld, int64_t cols_p, const double *shift,
                                   __nv_bfloat16 *hi, __nv_bfloat16 *lo, double *part,
                                   double *part_c, int first_chunk, cudaStream_t s);
// after the last chunk: delta_i = mu_i - s_i, ss, rs, and
// out[p] = (out[p] - D delta_i delta_j) rs_i rs_j
cudaError_t launch_slice_finalize(const double *part, const double *part_c, int64_t n,
                                  int64_t D, double *delta, double *ss, double *rs, double *out,
                                  cudaStream_t s);
cudaError_t launch_gram_f32(const float *C, int64_t n, int64_t Dp, const double *rs,
                            const int32_t *tiles, int64_t n_tiles, int32_t *queue, void *out,
                            int coverage, const double *delta, int64_t D, cudaStream_t s);
// tensor-core split-BF16 Gram (gram_tc.cu)
constexpr int kTcTileM = 128;    // rows of the I block per tile
constexpr int kTcTileN = 256;    // rows of the J block per tile
cudaError_t make_tc_tensor_maps(const __nv_bfloat16 *hi, const __nv_bfloat16 *lo,
                                int64_t n, int64_t Dp, void **tmap_hi, void **tmap_lo);
cudaError_t launch_gram_tc(const void *tmap_hi, const void *tmap_lo, int64_t n, int64_t Dp,
                           const double *rs, const int32_t *tiles, int64_t n_tiles,
                           int32_t *queue, int32_t *status, double *g64, void *out,
                           int coverage, int ooc, uint64_t budget, int32_t debug,
                           cudaStream_t s);
// split-BF16 Gram on CTA pairs (gram_tc2.cu): units of kOocTileInts int32
// {A row block of CTA 0, of CTA 1, B row block of CTA 0, of CTA 1, first row
// block (128 items) of the I block, J block (256 items), first chunk, end
// chunk}; atomic = 1 adds partial Grams into FP64 out, 0 writes G rs_i rs_j
// of whole block pairs, coverage = 1 counts pairs into int32 out.
cudaError_t launch_gram_tc2(const void *tmap_hi, const void *tmap_lo, int64_t n, const double *rs,
                            const int32_t *units, int64_t n_units, const UnitQueue &queue,
                            int32_t *status, double *g64, void *out, int coverage, int atomic,
                            uint64_t budget, int32_t debug, cudaStream_t s);
// split-K units of the resident set, listed by pair_units with k_split ranges
// of at most kKSplitCols columns: range r's partial Grams stored as FP32 in
// planes[r][n (n - 1) / 2]
cudaError_t launch_gram_tc2_store(const void *tmap_hi, const void *tmap_lo, int64_t n,
                                  const int32_t *units, int64_t n_units, int64_t k_split,
                                  const UnitQueue &queue, int32_t *status, float *planes,
                                  uint64_t budget, int32_t debug, cudaStream_t s);
// CTA pairs of one launch (clusters of two that fit on the device at once)
int64_t tc2_pairs();
// units of the CTA-pair Gram over the resident set: macro pairs (I <= J, 256
// items each) in recursive quadrant order, in waves of `group` macro pairs,
// k_split column ranges of the nchunks 64-column chunks per wave (k_split <= 1:
// one unit per macro pair over all columns)
void pair_units(int64_t n, int64_t nchunks, int64_t group, int64_t k_split,
                std::vector<int32_t> &units);
// the same for a given list of macro pairs (I, J) in the order to run them
void pair_units_of(const std::vector<int32_t> &macro_pairs, int64_t nchunks, int64_t group,
                   int64_t k_split, std::vector<int32_t> &units);
// out-of-core unit: {A row block, B row blocks (2), I block, J block, chunk
// begin, chunk end, unused}; chunks are 64 columns of D
constexpr int kOocTileInts = 8;
constexpr int kOocChunkCols = 64;
constexpr int kMaxKSplit = AP_MAX_K_SPLIT;
constexpr int64_t kKSplitCols = 16384;   // target columns per split-K unit
// CTAs of one Gram launch and the FP64 scratch (doubles) it needs: one
// 128 x 256 FP64 partial-sum tile per CTA
int64_t tc_grid(int64_t n_tiles);
size_t tc_scratch_doubles(int64_t n_tiles);
void free_tc_tensor_maps(void *tmap_hi, void *tmap_lo);
void tc_tiles(int64_t n, std::vector<int32_t> &tiles);   // (I-block of 128, J-block of 256)
// cloud tiles of a set whose points take under 16 MB: reordered largest
// first (point pairs per tile); returns whether it reordered
bool order_cloud_tiles(const std::vector<int32_t> &bstart, const std::vector<int64_t> &cnt,
                       int64_t total_pts, std::vector<int32_t> &tiles);
// split-K units of the tiles: waves of `group` tiles, column range-major
// inside each wave (k_split ranges of the nchunks 64-column chunks)
void panel_units(const std::vector<int32_t> &tiles, int64_t nchunks, int64_t group,
                 int64_t k_split, std::vector<int32_t> &units);
// the split-K schedule of a vector set's split-BF16 Gram: k_split column
// ranges per tile (0 whole tiles, -1 the default rule of default_k_split)
int32_t default_k_split(int64_t n_tiles, int64_t slots, int64_t Dp, int64_t pairs);
constexpr int64_t kPlaneBytes = 256ll << 20;    // most the planes of a set may take
ap_status set_vector_plan(ap_items *it, int32_t k_split, int32_t mma_ctas = 0);

// the particle scores' re-scaled cloud storage and L2 self terms, built on
// first use (api.cu)
ap_status ensure_score_storage(ap_items *it, int score, cudaStream_t s);
// pair lists (pairlist.cu): Pearson of listed pairs (host arrays) over the
// resident rows
cudaError_t launch_pearson_list(VecStore &v, bool split, const int32_t *pi,
                                const int32_t *pj, int64_t n_pairs, double *out,
                                cudaStream_t s);

// clouds (overlap.cu)
cudaError_t launch_overlap(const CloudStore &cs, const float *params, float *out,
                           int coverage, const UnitQueue &queue, cudaStream_t s);
// adjoint (params_io == NULL: grad_params = grad_out * grad f) or one fused
// ascent step (params_io != NULL: params_io += eta grad f / f where f >= fmin)
cudaError_t launch_overlap_grad_q(const CloudStore &cs, const UnitQueue &queue,
                                  const float *params, const float *grad_out,
                                  float *grad_params, float *f_out, float eta, float fmin,
                                  float *params_io, int32_t *flags, cudaStream_t s);
// particle scores (score 1 GMM L2 distance, 2 Bhattacharyya cost) on the
// re-scaled storage pts / lw; self = the L2 self terms (score 1)
cudaError_t launch_score(const CloudStore &cs, int score, const float4 *pts, const float *lw,
                         const double *self, const float *params, float *out,
                         const UnitQueue &queue, cudaStream_t s);
cudaError_t launch_cloud_rescore(const CloudStore &cs, int score, float4 *pts_out, float *lw_out,
                                 cudaStream_t s);
cudaError_t launch_cloud_self(const CloudStore &cs, const float4 *pts, const float *lw,
                              double *self, cudaStream_t s);
// sparse vectors (sparse.cu)
ap_status create_sparse(const ap_items_desc *d, ap_items *it, cudaStream_t s);
void free_sparse(SparseStore &sp);
cudaError_t launch_sparse_cosine(const SparseStore &sp, void *out, int coverage, cudaStream_t s);
constexpr int32_t kCloudWide = 1, kCloudWeighted = 2;   // traits of a set, see below
// tiles at the end of a cloud plan's list that are split: one per CTA slot
// (four CTAs of four warps per SM)
constexpr int64_t kSplitTailPerSm = 4;
constexpr int kOverlapMaxRows = 128;      // partial rows of a block of several items
constexpr int kOverlapMaxBlockItems = 32;
constexpr int kCloudStagePts = 2048;      // points of the staging buffer of a J block
cudaError_t launch_cloud_pack(const float *x, const float *y, const float *z,
                              const float *sigma, const float *w, const int64_t *src_off,
                              const int32_t *perm, const int64_t *poff, int64_t n, int dim,
                              float4 *pts, float *lw, float4 *boxes, bool boxed,
                              int64_t most_points, int32_t *traits, cudaStream_t s);

int num_sms();

// ---------------------------------------------------------------------------
// shared host helpers (api.cu, tune.cu)
// ---------------------------------------------------------------------------
ap_status from_cuda(cudaError_t e);
// propagate an ap_status
#define AP_TRY_ST(expr)                            \
  do {                                             \
    ap_status _s = (expr);                         \
    if (_s != AP_OK) return _s;                    \
  } while (0)

#define AP_TRY(expr)                               \
  do {                                             \
    cudaError_t _e = (expr);                       \
    if (_e != cudaSuccess) return ::ap::from_cuda(_e); \
  } while (0)
template <typename T>
cudaError_t dmalloc(T **p, size_t count) {
  *p = nullptr;
  if (count == 0) return cudaSuccess;
  return cudaMalloc(reinterpret_cast<void **>(p), count * sizeof(T));
}
template <typename T>
void dfree(T *&p) {
  if (p) cudaFree(reinterpret_cast<void *>(p));
  p = nullptr;
}

// A copy from pageable memory, and what the null stream was given before it, done
// for every stream on return.  cudaMemcpy by itself returns when the source has been
// staged, and a stream that does not wait for the null stream (a non-blocking
// one) may then read what was there before.
inline cudaError_t upload_now(void *dst, const void *src, size_t bytes) {
  const cudaError_t e = cudaMemcpy(dst, src, bytes, cudaMemcpyHostToDevice);
  return e == cudaSuccess ? cudaStreamSynchronize(nullptr) : e;
}

struct CloudPlanChoice { int32_t block_items, block_pts, reg_r; bool sorted; };
CloudPlanChoice choose_cloud_plan(const CloudStore &c);
ap_status build_cloud_plan(ap_items *it, const CloudPlanChoice &ch, cudaStream_t s);
// copy a plan to the device into c (its plan buffers hold nothing before)
ap_status upload_cloud_plan(CloudStore &c, const CloudPlanHost &h, cudaStream_t s);
void free_cloud_plan(CloudStore &c);
// per item of the set: {its block of one, 8 ints} as in CloudPlanHost::bmeta
void single_item_blocks(const CloudStore &c, int32_t reg_r, std::vector<int32_t> &bmeta);
// smallest a-points-per-lane that keeps the largest item within the row jobs
int32_t min_reg_r(const CloudStore &c);

// Launch `seq` on `s` through a cached CUDA graph captured on the handle's
// private stream (direct launch when `s` is itself being captured).
ap_status run_graphed(ap_items *it, const GraphKey &key, cudaStream_t s,
                      const std::function<cudaError_t(cudaStream_t)> &seq);
void clear_graphs(ap_items *it);

// out-of-core vector sets (slotcache.cu)
ap_status create_out_of_core(const ap_items_desc *d, ap_items *it);
ap_status run_out_of_core(ap_items *it, void *out, int coverage, cudaStream_t s);
void free_out_of_core(VecStore &v);
// host source streamed macro by macro into a resident set, each macro's pairs
// computed as soon as it is pre-processed (slotcache.cu)
ap_status stream_load_and_run(ap_items *it, const float *h, double *out, cudaStream_t s);

}  // namespace ap
