// overlap.cu -- Gaussian overlap cost between weighted point clouds, the
// cross term of the GMM L2 distance used by the microscopy application
// (Sec. V-C), its adjoint with respect to a rigid 2-D transform, and batched
// gradient ascent for pairwise registration.
//
//   f(i,j) = sum_a sum_b w_a w_b exp(-|x_a - (R x_b + t)|^2 / (2 (s_a^2 + s_b^2)))
//
// Storage (built by cloud_pack): items in planner order, padded to multiples
// of 4 points and held in pairs of points, s2k = 2 ln2 sigma^2 (negated) and
// lw = log2 w, so each term is
//   w_a * 2^(lw_b - d^2 / (s2k_a + s2k_b)).
// The FP32 work runs as packed FP32x2 operations on two b-points at a time.
// With a transform the a-points are moved instead of the b-points:
//   |x_a - (R x_b + t)| = |R^T (x_a - t) - x_b|,
// so the inner loop is unchanged, and the adjoint follows from
//   df/dt = 2 ln2 * R sum e r d',   df/dtheta = 2 ln2 * sum e r (x_b d'_y - y_b d'_x)
// with d' = R^T (x_a - t) - x_b and r = 1 / (s2k_a + s2k_b).
//
// The two particle scores of the microscopy application run through the same
// kernel (SCORE 1, 2) on re-scaled copies of the storage:
//   SCORE 1, GMM L2 cross term (s2k = 2 ln2 s^2, lw = log2 w):
//     term = w_a w_b (2 pi s2)^(-d/2) exp(-d^2 / (2 s2)) = C q^d 2^(lw_a + lw_b - d^2 q^2)
//   SCORE 2, Bhattacharyya (s2k = 4 ln2 s^2, lw = log2 w / 2 + (d/2) log2 sigma):
//     term = sqrt(w_a w_b) (2 s_a s_b / s2)^(d/2) exp(-d^2 / (4 s2)) = C q^d 2^(...)
// with q^2 = 1 / (s2k_a + s2k_b) and C = (ln2 / pi)^(d/2) or (8 ln2)^(d/2); the
// L2 distance adds the per-item self terms S_i + S_j - 2 C sum in the epilogue.
//
// Schedule: persistent CTAs take tiles (I block, J block) of the upper
// triangle of item blocks, the first by CTA index, the others from an atomic
// queue (Sec. IV-B), whose next tile is read while the current one is
// computed.  The J block's points are staged into shared memory as they lie
// with one bulk asynchronous copy per window; the CTA's warps take (job,
// partner item) units: a job is up to 128 a-points in registers, four per
// lane, of one large item or of pieces of several (see cloud_rows), swept
// against an item of J with broadcast shared-memory reads.  Each fragment's
// sum over its lanes does not depend on the job it shares, so a pair has the
// same bits in every plan of the same points per lane and in a pair list;
// its fragments meet in FP64 in order.
//
// What bounds the sweep (cycles per scheduler and warp of 2 x 32 terms, 2.06
// GHz): the FMA pipe, two cycles per packed operation (three where its three
// operands are distinct register pairs), with the MUFU's share beside it.  One
// reciprocal for two terms, 1/x = y / (x y), takes the overlap from 26.8 (the
// MUFU's 24 for two reciprocals and two exponentials) to 22.5, a third of
// which is the three extra products; the adjoint, where the FMA pipe is
// already the longer one, keeps its two reciprocals and loses 30.7 -> 27.8 by
// plain FMAs for its three-operand sums.  Measured before / after with the
// fragments that share warps and the split tail of the tile list: 256 2-D
// clouds of 64-128 points 197 / 119 us, 1000 lognormal 3-D clouds 50.8 / 41.2
// ms, the L2 score of 256 clouds of 1000-2000 points 27.2 / 22.1 ms (12.1 with
// the boxes of large sets, kBoxedMean), one adjoint step of 400 clouds of 100-400
// points 2.12 / 1.92 ms.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "ap_internal.h"

namespace ap {

namespace {

constexpr int kThreads = 128;
constexpr int kMaxBlockItems = kOverlapMaxBlockItems;
constexpr float kTwoLn2 = 1.3862943611198906f;

enum Mode { FWD = 0, FWD_T = 1, GRAD = 2, COVER = 3 };

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsq_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// a + b = {sum, rounding error} exactly (Knuth)
__device__ __forceinline__ float2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

// Padding points lie at x = kFar.  The points of a set that is swept without
// log-weights lie within kNear of 0 and have |s2k| <= kSharedMax: a point that
// its transform takes past 2 kNear has no term with them, but it might have one
// with the padding, so such points stop at kPark, from where they have neither.
constexpr float kFar = 1e18f, kNear = 1e15f, kPark = 5e17f;

// smallest / largest, NaN where an operand is one
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float warp_min(float x) {
  float r;
  asm("redux.sync.min.NaN.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float warp_max(float x) {
  float r;
  asm("redux.sync.max.NaN.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct TileCtx {
  int32_t t;               // tile index (n_tiles or more: none left)
  int32_t i_begin, i_end, j_begin, j_end;
  int32_t i_grp0, i_grps;  // groups of four storage points of the I block
  int32_t j_grp0, j_grps;
  int32_t job0, n_jobs;    // warp jobs of the I block
  int32_t diag;            // I block = J block
};

struct Params {
  const float4 *pts;
  const float *lw;
  const float4 *boxes;     // of the overlap's storage (see cloud_box0)
  const int4 *items;       // per stored item {first group, points, original id, first row}
  const int4 *bmeta;       // per block {item begin, end, first group, groups} {job0, jobs, rows, 0}
  const int2 *desc;        // [jobs][32] lane descriptors of blocks of several items
  const int32_t *tiles;
  int64_t n_tiles;
  int64_t n_items;
  int32_t *queue, *ahead;  // this launch's head, one it clears for another (or NULL)
  int32_t *status;
  const int32_t *traits;   // kCloudWide, kCloudWeighted
  int32_t stage_cap;       // points that fit the shared staging buffer (a multiple of 4)
  int32_t part_floats;     // partial sums of the largest tile
  int32_t list_mode;       // tiles are listed pairs: tile t's params and outputs
                           // sit at index t (not at the packed pair index)
  // outputs / extra inputs
  float *out;              // FWD: f[P]; COVER: int32 counts[P]
  const float *params;     // [P][3] (theta, tx, ty) or NULL
  const float *grad_out;   // [P] or NULL
  float *grad_params;      // [P][3]
  float *f_out;            // [P] or NULL
  float *params_io;        // ascent: params updated in place
  int32_t *flags;          // ascent: skipped steps
  float eta, fmin;
  const double *self;      // SCORE 1: S per original item
  double score_c;          // SCORE 1, 2: the constant C
};

// floats of one partial sum: f in two, the first and the last, and the adjoint's
// three components
template <int MODE>
constexpr int part_size() { return MODE == GRAD ? 5 : 2; }

// CTAs of four warps per SM that the registers must allow
template <int MODE>
constexpr int min_ctas() { return MODE == GRAD ? 3 : 4; }

// Items of up to kFewPoints take a reciprocal for each term.  A shared one puts
// three roundings where there was one, which the two-float sums make up for
// from dozens of terms on and not for a few: relative errors (rms) over pairs of
// clouds of 1 / 2 / 3 / 8 points 2.2e-7 / 7.8e-8 / 5.7e-8 / 4.5e-8 with it,
// 2.0e-7 / 7.2e-8 / 5.4e-8 / 4.4e-8 with one each (2-D).
// The choice costs 600 3-D clouds of 100-200 points 1.44 -> 1.47 ms, others less.
constexpr int kFewPoints = 8;

template <int DIM, int MODE, int R, int SCORE, bool BOX>
__global__ void __launch_bounds__(kThreads, min_ctas<MODE>())
overlap_kernel(Params P) {
  constexpr int NV = (MODE == GRAD) ? 4 : 1;     // partial values per (row, j)
  // a-points that a sum of f spans before it is held in two floats (as points, so
  // that a piece of up to 32 has the same bits whatever lanes it sits on)
  constexpr int kTwoFrom = MODE == GRAD ? 32 : 0;
  // Where neighbours are stored together, the adjoint's terms of one sign follow
  // one another and cancel late, so they are summed by blocks first (2-norm of the
  // gradient's error at 1500 points: 1.4e-7, 2.4e-7 in one sum, 1.75e-7 in one sum
  // over points as given).
  constexpr bool kBlockwise = MODE == GRAD && BOX;
  // The cost's terms of like size follow one another there too: they are added
  // two by two, in 3-D into blocks of 8 pairs.  Means over 24 lognormal sets of 50
  // to 5000 points, 2-norm: 3-D 5.52e-8 (one by one, blocks of 16 5.70e-8; points
  // as given, before the boxes 5.54e-8), 2-D 4.79e-8 (4.92e-8; 4.83e-8).  Two by
  // two is no slower (3-D 2% faster); with blocks of 8 and their exact addition
  // 1000 lognormal 3-D clouds take 40.7 ms, 40.0 before.
  constexpr bool kTree = BOX && SCORE == 0 && MODE != GRAD;
  constexpr int kFold = kTree && DIM == 3 ? 8 : 16;      // pairs of a block's sum
  constexpr int kPart = part_size<MODE>();       // floats per (row, j)
  constexpr int kUnroll = DIM == 3 ? 2 : 4;
  constexpr bool kRsq = SCORE != 0 && DIM == 3;  // terms need q^3: rsqrt, not a reciprocal
  extern __shared__ __align__(16) uint8_t smem[];
  float4 *s_pts = reinterpret_cast<float4 *>(smem);
  float2 *s_lw = reinterpret_cast<float2 *>(s_pts + P.stage_cap);
  float *s_part = reinterpret_cast<float *>(s_lw) + (DIM == 3 ? P.stage_cap : 0);
  // [32] item j's pairs in the window, first box (-1: no boxes), few points
  int4 *s_j = reinterpret_cast<int4 *>(s_part + P.part_floats);
  uint64_t *s_bar = reinterpret_cast<uint64_t *>(s_j + kMaxBlockItems);
  TileCtx *s_ctx = reinterpret_cast<TileCtx *>(s_bar + 1);       // [2] this tile, the next
  int *s_next = reinterpret_cast<int *>(s_ctx + 2);              // next (job, partner) unit

  const int lane = threadIdx.x & 31;
  const uint32_t bar = smem_u32(s_bar);
  uint32_t phase = 0;
  const int32_t traits = MODE == COVER ? 0 : __ldg(P.traits);
  const bool wide = (traits & kCloudWide) != 0;
  const bool plain = traits == 0 && SCORE != 2;   // SCORE 2's log-weights hold sigma

  // read a tile's blocks' ranges (thread 0; the chain of loads overlaps the
  // previous tile's arithmetic)
  auto fetch = [&](TileCtx *dst, int t) {
    if (*reinterpret_cast<volatile int32_t *>(P.status) != 0) t = (int)P.n_tiles;
    dst->t = t;
    if (t < P.n_tiles) {
      const int IB = P.tiles[2 * (int64_t)t], JB = P.tiles[2 * (int64_t)t + 1];
      const int4 a = P.bmeta[2 * (int64_t)IB], b = P.bmeta[2 * (int64_t)JB];
      const int4 jobs = P.bmeta[2 * (int64_t)IB + 1];
      dst->i_begin = a.x; dst->i_end = a.y; dst->i_grp0 = a.z; dst->i_grps = a.w;
      dst->j_begin = b.x; dst->j_end = b.y; dst->j_grp0 = b.z; dst->j_grps = b.w;
      dst->job0 = jobs.x; dst->n_jobs = jobs.y;
      dst->diag = !P.list_mode && b.x < a.y;
    }
  };
  // the first tile of a CTA is its index; each later pop takes the next
  auto pop = [&]() { return atomicAdd(P.queue, 1) + (int)gridDim.x; };
  if (threadIdx.x == 0) {
    if (blockIdx.x == 0 && P.ahead) *P.ahead = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fetch(s_ctx, blockIdx.x);
  }
  __syncthreads();

  for (int cur = 0;; cur ^= 1) {
    const TileCtx c = s_ctx[cur];
    if (c.t >= P.n_tiles) break;
    const int nJ = c.j_end - c.j_begin, nI = c.i_end - c.i_begin;
    const int j_pts = 4 * c.j_grps;
    if (MODE == COVER && threadIdx.x == 0) fetch(s_ctx + (cur ^ 1), pop());

    // the J block goes through the staging buffer at once, or an item larger than
    // that (a block by itself, so that every plan cuts it alike) in windows of
    // stage_cap points
    for (int w0 = 0; MODE != COVER && (w0 == 0 || w0 < j_pts); w0 += P.stage_cap) {
      const int w_pts = min(P.stage_cap, j_pts - w0);
      if (threadIdx.x == 0) {
        *s_next = 0;
        if (w_pts > 0) {
          // one bulk asynchronous copy per array, as the storage lies
          const int64_t p0 = 4 * (int64_t)c.j_grp0 + w0;
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          const uint32_t bytes = (uint32_t)w_pts * (DIM == 3 ? 20u : 16u);
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                       "r"(bytes)
                       : "memory");
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
                  "r"(smem_u32(s_pts)),
              "l"(P.pts + p0), "r"((uint32_t)(w_pts * 16)), "r"(bar)
              : "memory");
          if (DIM == 3)
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
                    "r"(smem_u32(s_lw)),
                "l"(P.lw + p0), "r"((uint32_t)(w_pts * 4)), "r"(bar)
                : "memory");
        }
      }
      for (int jl = threadIdx.x; jl < nJ; jl += blockDim.x) {
        const int4 m = __ldg(P.items + c.j_begin + jl);
        const int b0 = 4 * (m.x - c.j_grp0), b1 = b0 + m.y;
        const int q0 = max(b0, w0), q1 = min(b1, w0 + w_pts);
        const bool boxes = BOX && !wide && m.y > kCullPoints && ((q0 - b0) & 31) == 0;
        // up to one padding point, or (kTree) to the end of the last four
        const int end = kTree ? (q1 - w0 + 3) >> 2 << 1 : (q1 - w0 + 1) >> 1;
        s_j[jl] = make_int4((q0 - w0) >> 1, q1 > q0 ? end : (q0 - w0) >> 1,
                            boxes ? (int)cloud_box0(m.x, c.j_begin + jl) + (q0 - b0) / 32 : -1,
                            m.y <= kFewPoints);
      }
      __syncthreads();
      if (w0 == 0 && threadIdx.x == 0) fetch(s_ctx + (cur ^ 1), pop());
      if (w_pts > 0) {
        bool ok = true;
        uint32_t done = 0;
        const uint64_t t0 = global_ns();
        for (uint32_t it = 0;; ++it) {
          asm volatile(
              "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
              "selp.u32 %0, 1, 0, p;\n\t}"
              : "=r"(done)
              : "r"(bar), "r"(phase)
              : "memory");
          if (done) break;
          if ((it & 255u) == 255u && global_ns() - t0 > kWaitBudgetNs) { ok = false; break; }
        }
        phase ^= 1;
        if (!ok && threadIdx.x == 0) atomicCAS(P.status, 0, DEV_TIMEOUT_STAGE);
      }

      // One unit: a job's RE a-points per lane against item j.  Each lane's
      // points are part of one group of four storage points, so of one item.
      auto unit = [&](auto re, const int2 d, const int jl) {
        constexpr int RE = decltype(re)::value;
        const int row = d.y & 1023, t = (d.y >> 10) & 31, len = ((d.y >> 15) & 31) + 1;
        const int sub = (d.y >> 27) & 3;
        const bool active = d.x >= 0;
        // coordinates kept negated so d = b - a is one add, s2k as stored;
        // idle lanes and padding points have weight 0
        float ax[RE], ay[RE], az[RE], as[RE], aw[RE];
#pragma unroll
        for (int r = 0; r < RE; ++r) {
          ax[r] = ay[r] = az[r] = aw[r] = 0.f;
          as[r] = kRsq ? 1.f : -1.f;
        }
        if (active) {
#pragma unroll
          for (int p = 0; p < (RE + 1) / 2; ++p) {
            const int64_t pr = 2 * (int64_t)d.x + (RE == 4 ? p : RE == 2 ? sub : sub >> 1);
            const float4 u = __ldg(P.pts + 2 * pr), v = __ldg(P.pts + 2 * pr + 1);
            float2 l = make_float2(v.z, v.w);
            if (DIM == 3) l = __ldg(reinterpret_cast<const float2 *>(P.lw) + pr);
            if (RE == 1) {
              const bool h = sub & 1;
              ax[0] = -(h ? u.y : u.x);
              ay[0] = -(h ? u.w : u.z);
              if (DIM == 3) az[0] = -(h ? v.y : v.x);
              as[0] = DIM == 3 ? (h ? v.w : v.z) : (h ? v.y : v.x);
              aw[0] = exp2f(h ? l.y : l.x);
            } else {
              ax[2 * p] = -u.x; ax[(2 * p + 1) % RE] = -u.y;
              ay[2 * p] = -u.z; ay[(2 * p + 1) % RE] = -u.w;
              if (DIM == 3) { az[2 * p] = -v.x; az[(2 * p + 1) % RE] = -v.y; }
              as[2 * p] = DIM == 3 ? v.z : v.x;
              as[(2 * p + 1) % RE] = DIM == 3 ? v.w : v.y;
              aw[2 * p] = exp2f(l.x); aw[(2 * p + 1) % RE] = exp2f(l.y);
            }
          }
        }
        if (MODE == FWD_T || MODE == GRAD) {
          // -a' = R^T (-(x_a - t)) for the transform of this lane's pair (i, j)
          const float *pp = (MODE == GRAD && P.params_io) ? P.params_io : P.params;
          const int il = (d.y >> 20) & 31;
          // (a diagonal tile's lanes with i >= j have no pair)
          if (pp && active && !(c.diag && c.i_begin + il >= c.j_begin + jl)) {
            const int oi = __ldg(P.items + c.i_begin + il).z, oj = __ldg(P.items + c.j_begin + jl).z;
            const int64_t pidx = P.list_mode ? (int64_t)c.t
                                             : pair_index(oi < oj ? oi : oj, oi < oj ? oj : oi,
                                                          P.n_items);
            float sth, cth;
            const float ttx = pp[3 * pidx + 1], tty = pp[3 * pidx + 2];
            sincosf(pp[3 * pidx], &sth, &cth);
#pragma unroll
            for (int r = 0; r < RE; ++r) {
              const float ux = __fadd_rn(ax[r], ttx), uy = __fadd_rn(ay[r], tty);
              ax[r] = __fmaf_rn(cth, ux, __fmul_rn(sth, uy));
              ay[r] = __fmaf_rn(cth, uy, __fmul_rn(-sth, ux));
              if (plain && ax[r] < -kPark && ax[r] > -INFINITY) ax[r] = -kPark;
            }
          }
        }
        // the sweep over item j: each packed operation takes two b-points
        // against one a-point held in both halves
        float uY[RE], uT[RE];                    // kBlockwise: pY, pT of the blocks before
        const float2 z2 = make_float2(0.f, 0.f);
        float2 pF[RE], pC[RE], pY[RE], pT[RE];
#pragma unroll
        for (int r = 0; r < RE; ++r) {
          pF[r] = z2; pC[r] = z2; pY[r] = z2; pT[r] = z2;
          uY[r] = uT[r] = 0.f;
        }
        const int4 qr = s_j[jl];
        // Boxes: the lane's a-points that weigh anything, then the warp's, as
        // the sweep holds them (negated); b - a' is fl(b + (-a')), and rounding
        // keeps order, so the gap bounds every difference the sweep forms.
        // A warp with an a-point far out (or NaN, from its transform) sweeps
        // everything.
        float nx0, nx1, ny0, ny1, nz0 = 0.f, nz1 = 0.f, sa;
        const int n_blk = (qr.y - qr.x + 15) >> 4;
        bool boxed = qr.z >= 0;
        if (boxed) {
          nx0 = ny0 = nz0 = INFINITY;
          nx1 = ny1 = nz1 = -INFINITY;
          sa = 0.f;
#pragma unroll
          for (int r = 0; r < RE; ++r)
            if (aw[r] != 0.f) {
              nx0 = min_nan(nx0, ax[r]); nx1 = max_nan(nx1, ax[r]);
              ny0 = min_nan(ny0, ay[r]); ny1 = max_nan(ny1, ay[r]);
              if (DIM == 3) { nz0 = min_nan(nz0, az[r]); nz1 = max_nan(nz1, az[r]); }
              sa = fmaxf(sa, fabsf(as[r]));
            }
          nx0 = warp_min(nx0); nx1 = warp_max(nx1);
          ny0 = warp_min(ny0); ny1 = warp_max(ny1);
          if (DIM == 3) { nz0 = warp_min(nz0); nz1 = warp_max(nz1); }
          sa = warp_max(sa);
          boxed = nx0 > -kNear && nx1 < kNear && ny0 > -kNear && ny1 < kNear;
        }
        // of 32 blocks of 16 pairs from block `base`, those with a term that
        // may not be 0: 2^x rounds to 0 below -126 (subnormals flush), and
        // x <= log-weight - gap^2 / (s_a + s_b)
        auto live = [&](int base) -> uint32_t {
          const int left = n_blk - base;
          uint32_t mask = left >= 32 ? 0xffffffffu : (1u << left) - 1u;
          if (boxed) {
            bool on = false;
            if (lane < left) {
              const float4 u = __ldg(P.boxes + 2 * ((int64_t)qr.z + base + lane));
              const float4 v = __ldg(P.boxes + 2 * ((int64_t)qr.z + base + lane) + 1);
              const float gx = fmaxf(fmaxf(u.x + nx0, -(u.y + nx1)), 0.f);
              const float gy = fmaxf(fmaxf(u.z + ny0, -(u.w + ny1)), 0.f);
              float g2 = fmaf(gy, gy, gx * gx);
              if (DIM == 3) {
                const float gz = fmaxf(fmaxf(v.x + nz0, -(v.y + nz1)), 0.f);
                g2 = fmaf(gz, gz, g2);
              }
              float sb = v.z, l = v.w;
              if (SCORE == 2) {            // the score's own s2k and log-weight
                l = 0.5f * l + 0.25f * (float)DIM * __log2f(sb / kTwoLn2) + 0.01f;
                sb *= 2.f;
              }
              on = !(g2 > (127.f + l) * (sa + sb) * 1.0001f);
            }
            mask &= __ballot_sync(0xffffffffu, on);
          }
          return mask;
        };
        auto sweep = [&](auto plain_set, auto shared) {
          constexpr bool PLAIN = decltype(plain_set)::value;   // weights 1: no log-weight
          constexpr bool ONE = decltype(shared)::value && MODE != GRAD;
          auto block = [&](int qb, int qe) {
            float2 bF[RE];                  // this block's f terms (compensated below)
#pragma unroll
            for (int r = 0; r < RE; ++r) bF[r] = z2;
            // sum(r, e, -q^d) for each a-point's terms with pair q
            auto terms = [&](int q, auto sum) {
              const float4 u = s_pts[2 * q], v = s_pts[2 * q + 1];
              const float2 X = make_float2(u.x, u.y), Y = make_float2(u.z, u.w);
              const float2 S = DIM == 3 ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
              const float2 L = PLAIN ? z2 : DIM == 3 ? s_lw[q] : make_float2(v.z, v.w);
#pragma unroll
              for (int r = 0; r < RE; ++r) {
                const float2 dx = __fadd2_rn(X, make_float2(ax[r], ax[r]));          // b - a'
                const float2 dy = __fadd2_rn(Y, make_float2(ay[r], ay[r]));
                float2 d2 = __fmul2_rn(dx, dx);
                d2 = __ffma2_rn(dy, dy, d2);
                if (DIM == 3) {
                  const float2 dz = __fadd2_rn(make_float2(v.x, v.y), make_float2(az[r], az[r]));
                  d2 = __ffma2_rn(dz, dz, d2);
                }
                const float2 ns = __fadd2_rn(make_float2(as[r], as[r]), S);   // -s2k (kRsq: +)
                float2 nr, qd = z2;                                            // -1 / s2k
                if (kRsq) {
                  const float2 qq = make_float2(rsq_approx(ns.x), rsq_approx(ns.y));
                  nr = __fmul2_rn(qq, make_float2(-qq.x, -qq.y));
                  qd = __fmul2_rn(qq, nr);                                     // -q^3
                } else if (ONE) {
                  // one MUFU reciprocal for two terms: 1/x = y / (x y)
                  const float w = rcp_approx(__fmul_rn(ns.x, ns.y));
                  nr = make_float2(__fmul_rn(w, ns.y), __fmul_rn(w, ns.x));
                } else {
                  nr = make_float2(rcp_approx(ns.x), rcp_approx(ns.y));
                }
                // lw_b - d^2 / s2k
                const float2 arg = PLAIN ? __fmul2_rn(d2, nr) : __ffma2_rn(d2, nr, L);
                const float2 e = make_float2(ex2_approx(arg.x), ex2_approx(arg.y));
                sum(r, e, kRsq ? qd : nr);
                if (MODE == GRAD) {
                  // the gradient needs only u = sum -e r d' (d' = b - a'):
                  // df/dt ~ u and df/dtheta ~ nty u_x - ntx u_y, the b x b
                  // terms of sum e r (x_b d'_y - y_b d'_x) cancelling.  Four
                  // plain FMAs: a packed one with three distinct register
                  // pairs takes the pipe for more than two plain ones do.
                  const float2 ner = __fmul2_rn(e, nr);
                  pY[r].x = __fmaf_rn(ner.x, dx.x, pY[r].x);
                  pY[r].y = __fmaf_rn(ner.y, dx.y, pY[r].y);
                  pT[r].x = __fmaf_rn(ner.x, dy.x, pT[r].x);
                  pT[r].y = __fmaf_rn(ner.y, dy.y, pT[r].y);
                }
              }
            };
            if constexpr (kTree) {
#pragma unroll 1
              for (int q = qb; q < qe; q += 2) {         // (an even number of pairs)
                float2 e0[RE], e1[RE];
                terms(q, [&](int r, float2 e, float2) { e0[r] = e; });
                terms(q + 1, [&](int r, float2 e, float2) { e1[r] = e; });
#pragma unroll
                for (int r = 0; r < RE; ++r) bF[r] = __fadd2_rn(bF[r], __fadd2_rn(e0[r], e1[r]));
              }
            } else {
#pragma unroll kUnroll
              for (int q = qb; q < qe; ++q)
                terms(q, [&](int r, float2 e, float2 qd) {
                  bF[r] = SCORE ? __ffma2_rn(e, qd, bF[r]) : __fadd2_rn(bF[r], e);
                });
            }
#pragma unroll
            for (int r = 0; r < RE; ++r) {
              // compensated add of the block sum (each half on its own; pC =
              // minus the compensation)
              const float2 m1 = make_float2(-1.f, -1.f);
              if constexpr (kFold == 8) {
                // exact whichever is larger: a block of neighbours may outweigh
                // all that came before it
                const float2 tk = __fadd2_rn(pF[r], bF[r]), bb = __ffma2_rn(pF[r], m1, tk);
                const float2 ea = __ffma2_rn(__ffma2_rn(bb, m1, tk), m1, pF[r]);
                const float2 eb = __ffma2_rn(bb, m1, bF[r]);
                pC[r] = __fadd2_rn(pC[r], __fadd2_rn(ea, eb));
                pF[r] = tk;
              } else {
                const float2 yk = __fadd2_rn(bF[r], pC[r]);
                const float2 tk = __fadd2_rn(pF[r], yk);
                pC[r] = __fadd2_rn(yk, __ffma2_rn(tk, m1, pF[r]));
                pF[r] = tk;
              }
              if (kBlockwise) {
                uY[r] = __fadd_rn(uY[r], __fadd_rn(pY[r].x, pY[r].y));
                uT[r] = __fadd_rn(uT[r], __fadd_rn(pT[r].x, pT[r].y));
                pY[r] = z2;
                pT[r] = z2;
              }
            }
          };
          if (BOX) {
            for (int base = 0; base < n_blk; base += 32)
              for (uint32_t mask = live(base); mask; mask &= mask - 1) {
                const int qb = qr.x + 16 * (base + __ffs(mask) - 1), qe = min(qb + 16, qr.y);
                block(qb, min(qb + kFold, qe));
                if (kFold == 8 && qb + kFold < qe) block(qb + kFold, qe);
              }
          } else {
            for (int qb = qr.x; qb < qr.y; qb += 16) block(qb, min(qb + 16, qr.y));
          }
        };
        if (kRsq) {
          if (plain) sweep(std::true_type(), std::false_type());
          else sweep(std::false_type(), std::false_type());
        } else if (plain && (MODE == GRAD || !qr.w)) {
          sweep(std::true_type(), std::true_type());
        } else if (!wide && (MODE == GRAD || !qr.w)) {
          sweep(std::false_type(), std::true_type());
        } else {
          sweep(std::false_type(), std::false_type());
        }

        // The lane's points, then the lanes of a fragment, summed pairwise by
        // their place in the item (no contraction: every RE gives the same
        // bits), so a fragment's sum does not depend on the lanes it sits on.
        // Where two terms share a reciprocal (two more roundings a term), f is
        // carried as an unevaluated sum of two floats, which more than makes
        // up for them (256 clouds: 4.9e-8 off in the 2-norm, 5.9e-8 with plain
        // sums and a reciprocal each); 3% of a pass of 64-128 points, less of
        // larger items.  The adjoint's f is so from 32 points on, which makes up
        // for a fragment of 128 where 64 used to meet in FP64 (150 points: 5.9e-8,
        // 6.8e-8 with plain sums, 6.2e-8 with those of 64); 1.5% of an ascent step.
        float s[NV][RE], lo[RE];
#pragma unroll
        for (int r = 0; r < RE; ++r) {
          if (kTwoFrom == 0) {
            const float2 h = two_sum(pF[r].x, pF[r].y);
            s[0][r] = __fmul_rn(aw[r], h.x);
            lo[r] = __fmaf_rn(aw[r], __fadd_rn(h.y, __fadd_rn(pC[r].x, pC[r].y)),
                              __fmaf_rn(aw[r], h.x, -s[0][r]));
          } else {
            s[0][r] = __fmul_rn(aw[r], __fadd_rn(pF[r].x, pF[r].y));
            lo[r] = 0.f;
          }
          if (MODE == GRAD) {
            const float gx = kBlockwise ? uY[r] : __fadd_rn(pY[r].x, pY[r].y);
            const float gy = kBlockwise ? uT[r] : __fadd_rn(pT[r].x, pT[r].y);
            s[NV > 1 ? 1 : 0][r] = __fmul_rn(aw[r], gx);
            s[NV > 2 ? 2 : 0][r] = __fmul_rn(aw[r], gy);
            s[NV > 3 ? 3 : 0][r] =
                __fmul_rn(aw[r], __fmaf_rn(ay[r], gx, __fmul_rn(-ax[r], gy)));
          }
        }
        auto add2 = [](float &h, float &l, float h2, float l2) {
          const float2 t = two_sum(h, h2);
          h = t.x;
          l = __fadd_rn(t.y, __fadd_rn(l, l2));
        };
#pragma unroll
        for (int o = 1; o < RE; o <<= 1) {
#pragma unroll
          for (int r = 0; r < RE; r += 2 * o) {
            if (kTwoFrom == 0) add2(s[0][r], lo[r], s[0][r + o], lo[r + o]);
            else s[0][r] = __fadd_rn(s[0][r], s[0][r + o]);
#pragma unroll
            for (int q = 1; q < NV; ++q) s[q][r] = __fadd_rn(s[q][r], s[q][r + o]);
          }
        }
        float v[NV], vl = lo[0];
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q] = s[q][0];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const bool in = t + o < len;
          const float fh = __shfl_down_sync(0xffffffffu, v[0], o);
          if (o * RE >= kTwoFrom) {
            const float fl =
                o * RE > kTwoFrom || kTwoFrom == 0 ? __shfl_down_sync(0xffffffffu, vl, o) : 0.f;
            if (in) add2(v[0], vl, fh, fl);
          } else if (in) {
            v[0] = __fadd_rn(v[0], fh);
          }
#pragma unroll
          for (int q = 1; q < NV; ++q) {
            const float x = __shfl_down_sync(0xffffffffu, v[q], o);
            if (in) v[q] = __fadd_rn(v[q], x);
          }
        }
        if (active && t == 0) {
          float *dst = s_part + ((size_t)row * nJ + jl) * kPart;
          if (w0) {
            add2(v[0], vl, dst[0], dst[kPart - 1]);
#pragma unroll
            for (int q = 1; q < NV; ++q) v[q] = __fadd_rn(v[q], dst[q]);
          }
#pragma unroll
          for (int q = 0; q < NV; ++q) dst[q] = v[q];
          dst[kPart - 1] = vl;
        }
      };

      // warps take (job, partner item) units from a shared counter, so every
      // warp of the CTA runs until the window's work is gone
      for (;;) {
        int u = 0;
        if (lane == 0) u = atomicAdd(s_next, 1);
        u = __shfl_sync(0xffffffffu, u, 0);
        if (u >= c.n_jobs * nJ) break;
        const int k = u / nJ, jl = u - k * nJ;
        const int2 d = c.job0 >= 0 ? __ldg(P.desc + ((int64_t)c.job0 + k) * 32 + lane)
                                   : cloud_lane_desc(k, lane, c.i_grp0, c.i_grps, R, 0, 0);
        if (c.diag) {
          // j must follow some item of the job
          const int first = __reduce_min_sync(0xffffffffu, d.x >= 0 ? (d.y >> 20) & 31 : 32);
          if (c.j_begin + jl <= c.i_begin + first) continue;
        }
        if (w0 && s_j[jl].x >= s_j[jl].y) continue;        // item j is not in this window
        const int re = (d.y >> 25) & 3;
        if (R == 4 && re == 2) unit(std::integral_constant<int, R>(), d, jl);
        else if (re == 1) unit(std::integral_constant<int, 2>(), d, jl);
        else unit(std::integral_constant<int, 1>(), d, jl);
      }
      __syncthreads();
    }

    // each pair's partial rows in order, in FP64, then the stores
    for (int q = threadIdx.x; q < nI * nJ; q += blockDim.x) {
      const int il = q / nJ, jl = q - il * nJ;
      if (c.diag && c.j_begin + jl <= c.i_begin + il) continue;
      const int4 mi = __ldg(P.items + c.i_begin + il);
      const int oi = mi.z, oj = __ldg(P.items + c.j_begin + jl).z;
      const int64_t p =
          P.list_mode ? (int64_t)c.t : pair_index(oi < oj ? oi : oj, oi < oj ? oj : oi, P.n_items);
      if (MODE == COVER) {
        atomicAdd(reinterpret_cast<int32_t *>(P.out) + p, 1);
        continue;
      }
      double sF = 0.0, sX = 0.0, sY = 0.0, sT = 0.0;
      const int r0 = c.job0 >= 0 ? mi.w : 0, r1 = r0 + cloud_rows(mi.y, R);
      for (int row = r0; row < r1; ++row) {
        const float *src = s_part + ((size_t)row * nJ + jl) * kPart;
        // (a sum that left the FP32 range has no rounding error to add)
        sF += (double)src[0] + (isinf(src[0]) ? 0.0 : (double)src[kPart - 1]);
        if (MODE == GRAD) { sX += (double)src[1]; sY += (double)src[2]; sT += (double)src[3]; }
      }
      if (MODE == FWD || MODE == FWD_T) {
        // SCORE terms were summed with a negative factor
        if (SCORE == 1) P.out[p] = (float)(P.self[oi] + P.self[oj] + 2.0 * P.score_c * sF);
        else if (SCORE == 2) P.out[p] = (float)(-P.score_c * sF);
        else P.out[p] = (float)sF;
      } else if (MODE == GRAD) {
        // rotate the translation part back: df/dt = 2 ln2 R sum e r d'
        const float *pp = P.params_io ? P.params_io : P.params;
        float th = 0.f, ttx = 0.f, tty = 0.f;
        if (pp) { th = pp[3 * p]; ttx = pp[3 * p + 1]; tty = pp[3 * p + 2]; }
        float sth, cth;
        sincosf(th, &sth, &cth);
        const float f = (float)sF;
        const float gx = kTwoLn2 * (float)(cth * sX - sth * sY);
        const float gy = kTwoLn2 * (float)(sth * sX + cth * sY);
        const float gt = kTwoLn2 * (float)sT;
        if (P.f_out) P.f_out[p] = f;
        if (P.params_io) {
          // one ascent step on log f
          if (f >= P.fmin) {
            const float s = P.eta / f;
            P.params_io[3 * p] = th + s * gt;
            P.params_io[3 * p + 1] = ttx + s * gx;
            P.params_io[3 * p + 2] = tty + s * gy;
          } else if (P.flags) {
            P.flags[p] = 1;
          }
        } else {
          const float go = P.grad_out ? P.grad_out[p] : 1.f;
          P.grad_params[3 * p] = go * gt;
          P.grad_params[3 * p + 1] = go * gx;
          P.grad_params[3 * p + 2] = go * gy;
        }
      }
    }
    __syncthreads();
  }
}

// |s2k| in [2^-60, 2^59]: the product of two sums of s2k then stays normal,
// and so does its reciprocal, for the overlap's and the scores' scalings.
// Padding points lie far from every point of such a set, so that their terms
// are 0 without a log-weight (squared distances stay finite).
constexpr float kSharedMin = 8.6736174e-19f, kSharedMax = 5.7646075e17f;

// Pack one item per CTA into planner order, padded to a multiple of 4 points,
// in pairs (two per thread and trip), and its boxes.  Larger items are put in
// order first, so that 128 and 32 points in a row are near each other.  In 2-D
// sorted by y and cut into strips of whole warps' 128 points, each strip sorted
// by x (the sort-tile-recursive packing of R-trees: Leutenegger, Lopez and
// Edgington, 1997), each 64 points by y: strips of the extent, which leave a
// warp's points over two or three cells, kept more blocks (GMM L2 of 256 particles
// of 1000-2000 points 13.7 ms, now 12.1).  In 3-D rows of the extent, by x: blocks thin in x are
// passed over more often than cubes where items are cut once or twice an axis
// (strips by rank ran the lognormal set 1% slower).  Key and index are one
// word, sorted in shared memory (a bitonic network over the next power of two).
constexpr int kPackThreads = 256;
__global__ void __launch_bounds__(kPackThreads)
cloud_pack_kernel(const float *__restrict__ x, const float *__restrict__ y,
                  const float *__restrict__ z, const float *__restrict__ sigma,
                  const float *__restrict__ w, const int64_t *__restrict__ src_off,
                  const int32_t *__restrict__ perm, const int64_t *__restrict__ poff, int64_t n,
                  int dim, float4 *__restrict__ pts, float *__restrict__ lw,
                  float4 *__restrict__ boxes, bool boxed, int32_t *__restrict__ traits) {
  extern __shared__ uint32_t s_order[];            // [next power of two of the largest item]
  __shared__ float s_lo[3], s_hi[3], s_red[kPackThreads / 32][6];
  const double two_ln2 = 1.3862943611198906;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int32_t seen = 0;
  for (int64_t s = blockIdx.x; s < n; s += gridDim.x) {
    const int64_t o = perm[s];
    const int64_t src0 = src_off[o];
    const int cnt = (int)(src_off[o + 1] - src0);
    const int64_t q0 = poff[s] >> 1;
    const int pairs = (int)((poff[s + 1] - poff[s]) >> 1);
    const bool ordered = boxed && cnt > kCullPoints;
    if (ordered) {
      // the item's extent
      float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
      for (int k = tid; k < cnt; k += kPackThreads) {
        const float p[3] = {x[src0 + k], y[src0 + k], dim == 3 ? z[src0 + k] : 0.f};
#pragma unroll
        for (int d = 0; d < 3; ++d) { lo[d] = fminf(lo[d], p[d]); hi[d] = fmaxf(hi[d], p[d]); }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        for (int m = 16; m > 0; m >>= 1) {
          lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], m));
          hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], m));
        }
        if (lane == 0) { s_red[warp][d] = lo[d]; s_red[warp][3 + d] = hi[d]; }
      }
      __syncthreads();
      if (tid < 3) {
        float a = INFINITY, b = -INFINITY;
        for (int k = 0; k < kPackThreads / 32; ++k) {
          a = fminf(a, s_red[k][tid]);
          b = fmaxf(b, s_red[k][3 + tid]);
        }
        s_lo[tid] = a;
        s_hi[tid] = b;
      }
      __syncthreads();
      int m = 1;
      while (m < cnt) m <<= 1;
      for (int k = tid; k < m; k += kPackThreads) s_order[k] = k < cnt ? k : 0xffffffffu;
      // a coordinate's place in the item's extent, in 1 / n
      auto at = [&](uint32_t idx, int d, int n) -> int {
        const float lo = s_lo[d], e = s_hi[d] - lo;
        const float t = e > 0.f ? ((d == 0 ? x : d == 1 ? y : z)[src0 + idx] - lo) / e : 0.f;
        return t >= 0.f && t <= 1.f ? min((int)(t * (float)n), n - 1) : 0;   // (NaN, infinity)
      };
      // the order by key(place, index) of 17 bits, or that of runs of `run` places
      auto sort = [&](int run, auto key) {
        __syncthreads();
        for (int k = tid; k < cnt; k += kPackThreads) {
          const uint32_t idx = s_order[k] & 16383u;
          s_order[k] = (uint32_t)key(k, idx) << 14 | idx;
        }
        __syncthreads();
        for (int size = 2; size <= run; size <<= 1)
          for (int half = size >> 1; half > 0; half >>= 1) {
            for (int k = tid; k < m / 2; k += kPackThreads) {
              const int a = 2 * k - (k & (half - 1)), b = a + half;
              const uint32_t va = s_order[a], vb = s_order[b];
              if ((va > vb) == (size == run || (a & size) == 0)) {
                s_order[a] = vb;
                s_order[b] = va;
              }
            }
            __syncthreads();
          }
      };
      const float warps = ceilf((float)cnt / 128.f);
      if (dim == 3) {
        // rows of about 128 points a cube, walked back and forth (at most 25)
        const int cells = max(1, (int)rintf(cbrtf((float)cnt / 128.f)));
        sort(m, [&](int, uint32_t i) {
          const int zc = at(i, 2, cells), yc = at(i, 1, cells), xc = at(i, 0, 4096);
          const int row = zc * cells + ((zc & 1) ? cells - 1 - yc : yc);
          return row << 12 | ((row & 1) ? 4095 - xc : xc);
        });
      } else {
        // strips by rank (at most 11), each by x, 64 points by y
        const float cuts = fmaxf(1.f, rintf(sqrtf(warps)));
        const int strip = (int)ceilf(warps / cuts) * 128;
        sort(m, [&](int, uint32_t i) { return at(i, 1, 1 << 17); });
        sort(m, [&](int k, uint32_t i) { return k / strip << 10 | at(i, 0, 1024); });
        sort(64, [&](int, uint32_t i) { return at(i, 1, 1 << 17); });
      }
    }
    auto source = [&](int k) { return src0 + (ordered ? (int64_t)(s_order[k] & 16383u) : k); };
    for (int k = tid; k < pairs; k += kPackThreads) {
      // padding: far away, log-weight -inf
      float px[2] = {kFar, kFar}, py[2] = {0.f, 0.f}, pz[2] = {0.f, 0.f}, ps[2] = {-1.f, -1.f};
      float pl[2] = {-INFINITY, -INFINITY};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (2 * k + h >= cnt) continue;
        const int64_t a = source(2 * k + h);
        const double sg = (double)sigma[a];
        ps[h] = (float)(-two_ln2 * sg * sg);     // stored negated
        if (!(-ps[h] >= kSharedMin && -ps[h] <= kSharedMax)) seen |= kCloudWide;
        const float wt = w ? w[a] : 1.f;
        pl[h] = wt == 1.f ? 0.f : (wt > 0.f) ? (float)log2((double)wt) : -INFINITY;
        px[h] = x[a];
        py[h] = y[a];
        if (dim == 3) pz[h] = z[a];
        if (!(fabsf(px[h]) <= kNear && fabsf(py[h]) <= kNear && fabsf(pz[h]) <= kNear))
          seen |= kCloudWide;
        if (wt != 1.f) seen |= kCloudWeighted;
      }
      float4 *dst = pts + 2 * (q0 + k);
      dst[0] = make_float4(px[0], px[1], py[0], py[1]);
      if (dim == 3) {
        dst[1] = make_float4(pz[0], pz[1], ps[0], ps[1]);
        reinterpret_cast<float2 *>(lw)[q0 + k] = make_float2(pl[0], pl[1]);
      } else {
        dst[1] = make_float4(ps[0], ps[1], pl[0], pl[1]);
      }
    }
    if (ordered) {
      // one warp per box, a point per lane, as just stored (FP64, and log2 in
      // it, is slow here)
      __syncthreads();
      const int64_t b0 = cloud_box0(poff[s] >> 2, s);
      for (int b = warp; b * 32 < cnt; b += kPackThreads / 32) {
        const int k = b * 32 + lane, h = k & 1;
        float lo[3], hi[3], sm = 0.f, lm = -INFINITY;
#pragma unroll
        for (int d = 0; d < 3; ++d) { lo[d] = INFINITY; hi[d] = -INFINITY; }
        if (k < cnt) {
          const int64_t q = q0 + (k >> 1);
          const float4 u = pts[2 * q], v = pts[2 * q + 1];
          const float l = dim == 3 ? lw[2 * q + h] : h ? v.w : v.z;
          if (!(l == -INFINITY)) {                // others have no terms
            sm = fabsf(dim == 3 ? (h ? v.w : v.z) : (h ? v.y : v.x));
            lm = l;
            lo[0] = hi[0] = h ? u.y : u.x;
            lo[1] = hi[1] = h ? u.w : u.z;
            lo[2] = hi[2] = dim == 3 ? (h ? v.y : v.x) : 0.f;
          }
        }
        for (int m = 16; m > 0; m >>= 1) {
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], m));
            hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], m));
          }
          sm = fmaxf(sm, __shfl_xor_sync(0xffffffffu, sm, m));
          lm = fmaxf(lm, __shfl_xor_sync(0xffffffffu, lm, m));
        }
        if (lane == 0) {
          boxes[2 * (b0 + b)] = make_float4(lo[0], hi[0], lo[1], hi[1]);
          boxes[2 * (b0 + b) + 1] = make_float4(lo[2], hi[2], sm, lm);
        }
      }
    }
    __syncthreads();                             // before the order is replaced
  }
  if (seen) atomicOr(traits, seen);
}

// Re-scaled storage of a particle score from the overlap's storage
// (s2k = -2 ln2 sigma^2, lw = log2 w): SCORE 1 keeps both, SCORE 2 takes
// s2k = -4 ln2 sigma^2 and lw = lw / 2 + (d/4) log2 sigma^2; 3-D storage has
// s2k positive, since its terms take a square root.  Padding keeps lw = -inf.
__global__ void cloud_rescore_kernel(const float4 *__restrict__ pts, const float *__restrict__ lw,
                                     int64_t n_pairs, int dim, int score,
                                     float4 *__restrict__ out_pts, float *__restrict__ out_lw) {
  const float ln2x2 = 1.3862943611198906f;
  const float2 *l2 = reinterpret_cast<const float2 *>(lw);
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_pairs;
       k += (int64_t)gridDim.x * blockDim.x) {
    float4 q = pts[2 * k + 1];
    float2 s2k = dim == 3 ? make_float2(q.z, q.w) : make_float2(q.x, q.y);   // padding: -1
    float2 l = dim == 3 ? l2[k] : make_float2(q.z, q.w);
    if (score == 2) {
      // log2 of the mantissa and the exponent apart: one rounding of the size of l
      auto half = [&](float lw, float s) {
        int e;
        const float m = frexpf(-s / ln2x2, &e), d4 = 0.25f * (float)dim;
        return fmaf(d4, (float)e, fmaf(d4, log2f(m), 0.5f * lw));
      };
      l.x = half(l.x, s2k.x);
      l.y = half(l.y, s2k.y);
    }
    const float f = (score == 2 ? 2.f : 1.f) * (dim == 3 ? -1.f : 1.f);
    s2k.x *= f;
    s2k.y *= f;
    if (dim == 3) {
      q.z = s2k.x; q.w = s2k.y;
      reinterpret_cast<float2 *>(out_lw)[k] = l;
    } else {
      q = make_float4(s2k.x, s2k.y, l.x, l.y);
    }
    out_pts[2 * k] = pts[2 * k];
    out_pts[2 * k + 1] = q;
  }
}

// S_i = C sum over a, a' in item i of w_a w_a' q^d 2^(-d^2 q^2) (SCORE 1
// storage), one CTA per item, FP32 blocks of 8 terms folded into FP64
// (neighbours are stored together, so a block may hold many terms of one size).
template <int DIM>
__global__ void __launch_bounds__(256)
cloud_self_kernel(const float4 *__restrict__ pts, const float *__restrict__ lw,
                  const int64_t *__restrict__ poff, const int32_t *__restrict__ cnt,
                  const int32_t *__restrict__ perm, int64_t n, double c, double *__restrict__ S) {
  __shared__ double red[8];
  // {x, y, z, s2k > 0} and log-weight of storage point k
  auto point = [&](int64_t k, float &l) {
    const float4 u = pts[k & ~1ll], v = pts[(k & ~1ll) + 1];
    const bool h = k & 1;
    l = DIM == 3 ? lw[k] : (h ? v.w : v.z);
    return DIM == 3 ? make_float4(h ? u.y : u.x, h ? u.w : u.z, h ? v.y : v.x, h ? v.w : v.z)
                    : make_float4(h ? u.y : u.x, h ? u.w : u.z, 0.f, h ? -v.y : -v.x);
  };
  for (int64_t it = blockIdx.x; it < n; it += gridDim.x) {
    const int64_t p0 = poff[it];
    const int m = cnt[it];
    double acc = 0.0;
    for (int a = threadIdx.x; a < m; a += blockDim.x) {
      float la, lb;
      const float4 qa = point(p0 + a, la);
      float part = 0.f;
      for (int b = 0; b < m; ++b) {
        const float4 qb = point(p0 + b, lb);
        const float dx = qb.x - qa.x, dy = qb.y - qa.y;
        float d2 = fmaf(dx, dx, dy * dy);
        if (DIM == 3) {
          const float dz = qb.z - qa.z;
          d2 = fmaf(dz, dz, d2);
        }
        const float q = rsq_approx(qa.w + qb.w), r = q * q;
        const float e = ex2_approx(fmaf(-d2, r, la + lb));
        part = fmaf(e, DIM == 2 ? r : r * q, part);
        if ((b & 7) == 7) { acc += widen(part); part = 0.f; }
      }
      acc += (double)part;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double tot = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
      S[perm[it]] = c * tot;
    }
    __syncthreads();
  }
}

template <int DIM, int MODE, int SCORE = 0>
cudaError_t launch_r(const CloudStore &cs, const UnitQueue &queue, Params &P, cudaStream_t s) {
  constexpr int kPart = part_size<MODE>();
  P.stage_cap = MODE == COVER ? 0 : (std::min(cs.max_pts, kCloudStagePts) + 3) & ~3;
  P.part_floats = MODE == COVER ? 0 : ((cs.max_rows * cs.max_items * kPart + 3) & ~3);
  const size_t smem = (size_t)P.stage_cap * (DIM == 3 ? 20 : 16) + (size_t)P.part_floats * 4 +
                      kMaxBlockItems * sizeof(int4) + 8 + 2 * sizeof(TileCtx) + 16;
  void (*kern)(Params) = cs.reg_r == 2 ? overlap_kernel<DIM, MODE, 2, SCORE, false>
                         : cs.boxed && MODE != COVER
                             ? overlap_kernel<DIM, MODE, 4, SCORE, MODE != COVER>
                             : overlap_kernel<DIM, MODE, 4, SCORE, false>;
  // listed pairs are tiles of one item against one, a few jobs each: one
  // warp per CTA and many CTAs per SM keep the warps busy (20 ascent steps on
  // 131K listed pairs: 114 ms at 8 warps per CTA, 89 at 4, 81 at 2, 79 at 1)
  const int threads = cs.list_mode ? 32 : kThreads;
  // the attribute and the CTAs that fit are looked up once per plan: the two
  // calls take as long as a launch
  int64_t slots = 0;
  for (const CloudStore::Fit &f : *cs.fits)
    if (f.kern == reinterpret_cast<const void *>(kern) && f.smem == smem && f.threads == threads)
      slots = f.slots;
  cudaError_t e = cudaSuccess;
  if (slots == 0) {
    // (the attribute is the kernel's, not the handle's: always the most a CTA
    // may have, so that no handle lowers it for another)
    int optin = 0, dev = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
      e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    int per_sm = 0;
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e != cudaSuccess) return leave_queue(queue, s, e);
    slots = (int64_t)num_sms() * std::max(per_sm, 1);
    cs.fits->push_back({reinterpret_cast<const void *>(kern), smem, threads, slots});
  }
  const int64_t grid = std::min(slots, P.n_tiles);
  kern<<<(int)grid, threads, smem, s>>>(P);
  e = cudaGetLastError();
  return e == cudaSuccess ? e : leave_queue(queue, s, e);
}

Params base_params(const CloudStore &cs, const UnitQueue &queue) {
  Params P{};
  P.pts = cs.d_pts;
  P.lw = cs.d_lw;
  P.boxes = cs.d_boxes;
  P.items = reinterpret_cast<const int4 *>(cs.d_items);
  P.bmeta = reinterpret_cast<const int4 *>(cs.d_bmeta);
  P.desc = reinterpret_cast<const int2 *>(cs.d_desc);
  P.tiles = cs.d_tiles;
  P.n_tiles = cs.n_tiles;
  P.n_items = cs.n;
  P.queue = queue.head;
  P.ahead = queue.ahead;
  P.status = queue.words + 1;
  P.traits = queue.words + kQueueTraits;
  P.list_mode = cs.list_mode ? 1 : 0;
  return P;
}

}  // namespace

cudaError_t launch_overlap(const CloudStore &cs, const float *params, float *out, int coverage,
                           const UnitQueue &queue, cudaStream_t s) {
  if (cs.n_tiles <= 0) return leave_queue(queue, s, cudaSuccess);
  Params P = base_params(cs, queue);
  P.out = out;
  P.params = params;
  if (coverage)
    return cs.dim == 3 ? launch_r<3, COVER>(cs, queue, P, s) : launch_r<2, COVER>(cs, queue, P, s);
  if (params) return launch_r<2, FWD_T>(cs, queue, P, s);
  return cs.dim == 3 ? launch_r<3, FWD>(cs, queue, P, s) : launch_r<2, FWD>(cs, queue, P, s);
}

cudaError_t launch_score(const CloudStore &cs, int score, const float4 *pts, const float *lw,
                         const double *self, const float *params, float *out,
                         const UnitQueue &queue, cudaStream_t s) {
  if (cs.n_tiles <= 0) return leave_queue(queue, s, cudaSuccess);
  Params P = base_params(cs, queue);
  P.pts = pts;
  P.lw = lw;
  P.out = out;
  P.params = params;
  P.self = self;
  P.score_c = score == 1 ? pow(0.6931471805599453 / 3.141592653589793, 0.5 * cs.dim)
                         : pow(8.0 * 0.6931471805599453, 0.5 * cs.dim);
  if (score == 1) {
    if (params) return launch_r<2, FWD_T, 1>(cs, queue, P, s);
    return cs.dim == 3 ? launch_r<3, FWD, 1>(cs, queue, P, s) : launch_r<2, FWD, 1>(cs, queue, P, s);
  }
  if (params) return launch_r<2, FWD_T, 2>(cs, queue, P, s);
  return cs.dim == 3 ? launch_r<3, FWD, 2>(cs, queue, P, s) : launch_r<2, FWD, 2>(cs, queue, P, s);
}

cudaError_t launch_cloud_rescore(const CloudStore &cs, int score, float4 *pts_out, float *lw_out,
                                 cudaStream_t s) {
  if (cs.total_pts <= 0) return cudaSuccess;
  const int64_t pairs = cs.total_pts / 2, blocks = (pairs + 255) / 256;
  cloud_rescore_kernel<<<(int)(blocks < 65535 ? blocks : 65535), 256, 0, s>>>(
      cs.d_pts, cs.d_lw, pairs, cs.dim, score, pts_out, lw_out);
  return cudaGetLastError();
}

cudaError_t launch_cloud_self(const CloudStore &cs, const float4 *pts, const float *lw,
                              double *self, cudaStream_t s) {
  if (cs.n <= 0) return cudaSuccess;
  const double c = pow(0.6931471805599453 / 3.141592653589793, 0.5 * cs.dim);
  const int grid = (int)(cs.n < 65535 ? cs.n : 65535);
  if (cs.dim == 3)
    cloud_self_kernel<3><<<grid, 256, 0, s>>>(pts, lw, cs.d_poff, cs.d_cnt, cs.d_perm, cs.n, c,
                                              self);
  else
    cloud_self_kernel<2><<<grid, 256, 0, s>>>(pts, lw, cs.d_poff, cs.d_cnt, cs.d_perm, cs.n, c,
                                              self);
  return cudaGetLastError();
}

cudaError_t launch_overlap_grad_q(const CloudStore &cs, const UnitQueue &queue,
                                  const float *params, const float *grad_out,
                                  float *grad_params, float *f_out, float eta, float fmin,
                                  float *params_io, int32_t *flags, cudaStream_t s) {
  if (cs.n_tiles <= 0) return leave_queue(queue, s, cudaSuccess);
  Params P = base_params(cs, queue);
  P.params = params;
  P.grad_out = grad_out;
  P.grad_params = grad_params;
  P.f_out = f_out;
  P.params_io = params_io;
  P.flags = flags;
  P.eta = eta;
  P.fmin = fmin;
  return launch_r<2, GRAD>(cs, queue, P, s);
}

cudaError_t launch_cloud_pack(const float *x, const float *y, const float *z, const float *sigma,
                              const float *w, const int64_t *src_off, const int32_t *perm,
                              const int64_t *poff, int64_t n, int dim, float4 *pts, float *lw,
                              float4 *boxes, bool boxed, int64_t most_points,
                              int32_t *traits, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  // (up to 64 KB: 16384 points, always allowed, so that no call lowers it)
  cudaError_t e = cudaFuncSetAttribute(cloud_pack_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, 16384 * 4);
  if (e != cudaSuccess) return e;
  int64_t m = 1;
  while (m < most_points) m <<= 1;
  const size_t smem = boxed && most_points > kCullPoints ? (size_t)m * 4 : 0;
  const int grid = (int)(n < 65535 ? n : 65535);
  cloud_pack_kernel<<<grid, kPackThreads, smem, s>>>(x, y, z, sigma, w, src_off, perm, poff, n, dim,
                                                     pts, lw, boxes, boxed, traits);
  return cudaGetLastError();
}

}  // namespace ap
