// pairlist.cu -- the pair function over a chosen list of pairs instead of the
// whole upper triangle: the comparison stage of Sec. III on a subset, and the
// per-pair registration of chosen pairs (Sec. V-C).
//
// Clouds reuse the all-pairs kernel: each listed pair (a, b) becomes a tile
// of two one-item blocks (storage positions of a and b), and the kernel's
// list mode puts tile t's transform and outputs at index t; the transform
// acts on b, as it acts on the second item of a packed pair.  A pair listed
// in packed order (a < b) therefore gets exactly the operations, and the
// bits, of the all-pairs run (of a plan of the same points per lane).
//
// Vectors run over the resident centred rows (split BF16 or FP32 copy), the
// same three products per column as the tensor-core Gram, summed in FP32 over
// 64 columns per lane and in FP64 after:
//   r_k = (sum_c c_a c_b - D delta_a delta_b) rs_a rs_b.
// The list runs in column slices that the rows it touches share in L2, and
// pairs with a row in common are computed together by one warp.
// Sparse rows merge their sorted codes (one CTA per pair).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "ap_internal.h"

namespace ap {

namespace {

constexpr int kListThreads = 256;

// Vector pairs.  Work is (column slice, group): a group is a row a and up to
// kListGroup partner rows, one warp's; the slices come one after another, so
// that the warps in flight read one slice of the touched rows, which stays in
// L2: a row's pieces (64 bytes, 8 KB apart) come from memory about once, not
// once per pair.  Bound by the L2 reads of the groups' rows.  3000 random pairs of
// 1024 x 2^18 (1 GiB of rows, 6.3 GB listed, 4.2 GB after grouping): 0.62 ms
// against 1.33 through a row-major copy of the touched blocks; 441 pairs of 389
// x 139,141, which read the pieces once per pair before: 65 us against 668.
// Slices of 12 and 40 MB and groups of 6 took as long, 6 MB 14% and groups of 8
// (spilled) 70% longer; asking for the next slice's blocks ahead 6% longer.
constexpr int kListGroup = 4;
constexpr int64_t kListSliceBytes = 24ll << 20;  // of the touched rows

struct ListPlan {
  const int4 *groups;        // {a, first pair, pairs, 0}
  const int32_t *a, *b;      // rows of the pairs in group order
  const int32_t *pos;        // their places in the caller's list
  int64_t n_groups, n_pairs, slice_cols, n_slices;
};

template <bool SPLIT>
__global__ void __launch_bounds__(kListThreads)
pearson_list_kernel(const __nv_bfloat16 *__restrict__ hi, const __nv_bfloat16 *__restrict__ lo,
                    const float *__restrict__ c32, int64_t Dp, ListPlan L,
                    double *__restrict__ part) {
  constexpr int kblk = SPLIT ? kTcKBlock : kF32KBlock;             // columns of an 8 KB block
  constexpr int64_t kBlock = (int64_t)kRowBlock * kblk;            // its elements
  constexpr int kCols = SPLIT ? 8 : 4;                             // columns of a 16-byte load
  constexpr int kTrip = 32 * kCols;                                // of a warp's trip
  const int lane = threadIdx.x & 31;
  const int64_t nkb = Dp / kblk;
  const int64_t per_slice = (L.n_groups + kListThreads / 32 - 1) / (kListThreads / 32);
  for (int64_t unit = blockIdx.x; unit < per_slice * L.n_slices; unit += gridDim.x) {
    const int64_t s = unit / per_slice, cta = unit - s * per_slice;
    const int64_t c0 = s * L.slice_cols, c1 = c0 + L.slice_cols < Dp ? c0 + L.slice_cols : Dp;

    const int64_t gi = cta * (kListThreads / 32) + (threadIdx.x >> 5);
    if (gi >= L.n_groups) continue;
    const int4 g = L.groups[gi];
    // a lane's first columns: load q of a trip covers block (q, lane >> 2)
    const int64_t k0 = c0 / kblk + (lane >> 2);
    auto at = [&](int64_t row) {
      return ((row / kRowBlock) * nkb + k0) * kBlock + (row % kRowBlock) * kblk + (lane & 3) * kCols;
    };
    int64_t oa = at(g.x), ob[kListGroup];
#pragma unroll
    for (int j = 0; j < kListGroup; ++j) ob[j] = at(L.b[g.y + (j < g.z ? j : 0)]);
    float sum[kListGroup];
    double acc[kListGroup];
#pragma unroll
    for (int j = 0; j < kListGroup; ++j) {
      sum[j] = 0.f;
      acc[j] = 0.0;
    }
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    auto load = [](const void *p, bool in) {
      return in ? __ldg(reinterpret_cast<const uint4 *>(p)) : make_uint4(0u, 0u, 0u, 0u);
    };
    int trips = 0;
    for (int64_t c = c0; c < c1; c += kTrip) {
      const bool in = c + (lane >> 2) * kblk < c1;
      uint4 ah, al = z, bh[kListGroup], bl[kListGroup];
      if (SPLIT) {
        ah = load(hi + oa, in);
        al = load(lo + oa, in);
      } else {
        ah = load(c32 + oa, in);
      }
#pragma unroll
      for (int j = 0; j < kListGroup; ++j) {
        bl[j] = z;
        bh[j] = z;
        if (j >= g.z) continue;
        if (SPLIT) {
          bh[j] = load(hi + ob[j], in);
          bl[j] = load(lo + ob[j], in);
        } else {
          bh[j] = load(c32 + ob[j], in);
        }
      }
      const uint32_t ahw[4] = {ah.x, ah.y, ah.z, ah.w}, alw[4] = {al.x, al.y, al.z, al.w};
#pragma unroll
      for (int j = 0; j < kListGroup; ++j) {
        if (j >= g.z) continue;
        const uint32_t bhw[4] = {bh[j].x, bh[j].y, bh[j].z, bh[j].w};
        const uint32_t blw[4] = {bl[j].x, bl[j].y, bl[j].z, bl[j].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (SPLIT) {
#pragma unroll
            for (int w = 0; w < 2; ++w) {            // the word's low and high bf16
              auto f = [&](uint32_t x) { return __uint_as_float(w ? x & 0xffff0000u : x << 16); };
              sum[j] = fmaf(f(ahw[e]), f(bhw[e]), sum[j]);
              sum[j] = fmaf(f(ahw[e]), f(blw[e]), sum[j]);
              sum[j] = fmaf(f(alw[e]), f(bhw[e]), sum[j]);
            }
          } else {
            sum[j] = fmaf(__uint_as_float(ahw[e]), __uint_as_float(bhw[e]), sum[j]);
          }
        }
      }
      oa += (int64_t)(kTrip / kblk) * kBlock;
#pragma unroll
      for (int j = 0; j < kListGroup; ++j) ob[j] += (int64_t)(kTrip / kblk) * kBlock;
      if (++trips == 64 / kCols) {                   // 64 columns per lane
        trips = 0;
#pragma unroll
        for (int j = 0; j < kListGroup; ++j) {
          acc[j] += widen(sum[j]);
          sum[j] = 0.f;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kListGroup; ++j) {
      if (j >= g.z) continue;
      double v = acc[j] + widen(sum[j]);
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) part[s * L.n_pairs + g.y + j] = v;
    }
  }
}

// the slices' sums in order, the mean correction and the scaling
__global__ void pearson_list_sum_kernel(const double *__restrict__ part, ListPlan L,
                                        const double *__restrict__ rs,
                                        const double *__restrict__ delta, int64_t D,
                                        double *__restrict__ out) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < L.n_pairs;
       q += (int64_t)gridDim.x * blockDim.x) {
    double g = 0.0;
#pragma unroll 8
    for (int64_t s = 0; s < L.n_slices; ++s) g += part[s * L.n_pairs + q];
    const int64_t a = L.a[q], b = L.b[q];
    out[L.pos[q]] = (g - (double)D * delta[a] * delta[b]) * rs[a] * rs[b];
  }
}

// Sparse rows (strictly increasing codes): one CTA per listed pair, each
// thread merging an even slice of row a's entries against row b from the
// first code of b at or after its slice (a binary search), so a pair costs
// about nnz_a + nnz_b reads; FP32 products summed per thread in FP64.
constexpr int kMergeThreads = 256;
__global__ void __launch_bounds__(kMergeThreads)
cosine_list_kernel(const int64_t *__restrict__ off, const int32_t *__restrict__ idx,
                   const float *__restrict__ val, const double *__restrict__ rs,
                   const int32_t *__restrict__ pi, const int32_t *__restrict__ pj,
                   int64_t n_pairs, double *__restrict__ out) {
  __shared__ double red[kMergeThreads / 32];
  for (int64_t k = blockIdx.x; k < n_pairs; k += gridDim.x) {
    const int64_t a = pi[k], b = pj[k];
    const int64_t a0 = off[a], na = off[a + 1] - a0, b0 = off[b], nb = off[b + 1] - b0;
    const int64_t per = (na + blockDim.x - 1) / blockDim.x;
    const int64_t s0 = (int64_t)threadIdx.x * per, s1 = s0 + per < na ? s0 + per : na;
    double acc = 0.0;
    if (s0 < s1) {
      // first entry of b whose code is >= the slice's first code
      const int32_t c0 = idx[a0 + s0];
      int64_t lo = 0, hi = nb;
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (idx[b0 + mid] < c0) lo = mid + 1;
        else hi = mid;
      }
      int64_t q = lo;
      for (int64_t e = s0; e < s1 && q < nb; ++e) {
        const int32_t code = idx[a0 + e];
        while (q < nb && idx[b0 + q] < code) ++q;
        if (q < nb && idx[b0 + q] == code) acc += (double)(val[a0 + e] * val[b0 + q]);
      }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
      out[k] = t * rs[a] * rs[b];
    }
    __syncthreads();
  }
}

// host checks shared by every list call: indices in range, a != b
ap_status check_list(const ap_items *it, const int32_t *pi, const int32_t *pj, int64_t n_pairs,
                     int64_t n) {
  if (n_pairs < 0 || (n_pairs > 0 && (!pi || !pj))) return AP_ERR_INVALID_ARG;
  if (n_pairs > INT32_MAX) return AP_ERR_UNSUPPORTED;   // tile indices are int32
  for (int64_t k = 0; k < n_pairs; ++k)
    if (pi[k] < 0 || pj[k] < 0 || pi[k] >= n || pj[k] >= n || pi[k] == pj[k])
      return AP_ERR_INVALID_ARG;
  (void)it;
  return AP_OK;
}

// the temporary list plan of a cloud set: one-item blocks, the listed pairs
// as tiles (storage positions), copied to the handle's list buffer on `s`
ap_status cloud_list_plan(ap_items *it, const int32_t *pi, const int32_t *pj, int64_t n_pairs,
                          cudaStream_t s, CloudStore &lc) {
  CloudStore &c = it->cl;
  if (c.h_iperm.size() != (size_t)c.n) {
    c.h_iperm.assign((size_t)c.n, 0);
    for (int64_t p = 0; p < c.n; ++p) c.h_iperm[c.h_perm[p]] = (int32_t)p;
  }
  if (!c.d_bmeta_single) {
    std::vector<int32_t> single;
    single_item_blocks(c, c.reg_r, single);
    AP_TRY(dmalloc(&c.d_bmeta_single, std::max<size_t>(single.size(), 8)));
    AP_TRY(upload_now(c.d_bmeta_single, single.data(), single.size() * 4));
  }
  if (c.list_cap < n_pairs) {
    AP_TRY(cudaStreamSynchronize(s));              // the old list may still be read
    dfree(c.d_list_tiles);
    c.list_cap = 0;
    AP_TRY(dmalloc(&c.d_list_tiles, (size_t)n_pairs * 2));
    c.list_cap = n_pairs;
  } else {
    AP_TRY(cudaStreamSynchronize(s));
  }
  std::vector<int32_t> tiles((size_t)n_pairs * 2);
  for (int64_t k = 0; k < n_pairs; ++k) {
    tiles[2 * k] = c.h_iperm[pi[k]];
    tiles[2 * k + 1] = c.h_iperm[pj[k]];
    // sets stored by size (3-D, without transforms): as the all-pairs run takes
    // them, the earlier in the storage first
    if (c.sorted && tiles[2 * k] > tiles[2 * k + 1]) std::swap(tiles[2 * k], tiles[2 * k + 1]);
  }
  // (a pageable source: staged before the call returns)
  AP_TRY(cudaMemcpyAsync(c.d_list_tiles, tiles.data(), tiles.size() * 4, cudaMemcpyHostToDevice, s));
  lc = c;
  lc.list_mode = true;
  lc.d_bmeta = c.d_bmeta_single;
  lc.d_tiles = c.d_list_tiles;
  lc.n_tiles = n_pairs;
  lc.max_items = lc.max_rows = 1;
  lc.max_pts = 4;
  for (int64_t p = 0; p < c.n; ++p) {
    lc.max_rows = std::max(lc.max_rows, cloud_rows(c.h_size[c.h_perm[p]], c.reg_r));
    lc.max_pts = std::max(lc.max_pts, (int32_t)(c.h_poff[p + 1] - c.h_poff[p]));
  }
  return AP_OK;
}

// the listed pairs' indices on the device (host arrays in, stream-ordered)
ap_status device_pairs(const int32_t *pi, const int32_t *pj, int64_t n_pairs, cudaStream_t s,
                       int32_t **d_idx) {
  AP_TRY(dmalloc(d_idx, (size_t)n_pairs * 2));
  AP_TRY(cudaMemcpyAsync(*d_idx, pi, (size_t)n_pairs * 4, cudaMemcpyHostToDevice, s));
  AP_TRY(cudaMemcpyAsync(*d_idx + n_pairs, pj, (size_t)n_pairs * 4, cudaMemcpyHostToDevice, s));
  return AP_OK;
}

// The listed vector pairs in groups that share a row: each pair goes to the
// end listed more often (r is symmetric), the pairs of a row in groups of up
// to kListGroup.  Host arrays for one copy: [groups x 4][a][b][position].
struct ListHost {
  std::vector<int32_t> ints;
  int64_t n_groups = 0, n_rows = 0;
};
void group_pairs(const int32_t *pi, const int32_t *pj, int64_t n_pairs, int64_t n, ListHost &h) {
  // the rows listed, numbered; their counts
  std::vector<int32_t> count((size_t)n, 0), first((size_t)n + 1, 0);
  for (int64_t k = 0; k < n_pairs; ++k) {
    ++count[pi[k]];
    ++count[pj[k]];
  }
  auto hub = [&](int64_t k) {
    return count[pj[k]] > count[pi[k]] || (count[pj[k]] == count[pi[k]] && pj[k] < pi[k]) ? pj[k]
                                                                                            : pi[k];
  };
  for (int64_t k = 0; k < n_pairs; ++k) ++first[hub(k) + 1];
  for (int64_t i = 0; i < n; ++i) {
    h.n_groups += (first[i + 1] + kListGroup - 1) / kListGroup;
    h.n_rows += count[i] > 0;
    first[i + 1] += first[i];
  }
  h.ints.resize((size_t)(4 * h.n_groups + 3 * n_pairs));
  int32_t *g = h.ints.data(), *a = g + 4 * h.n_groups, *b = a + n_pairs, *pos = b + n_pairs;
  for (int64_t i = 0; i < n; ++i)
    for (int32_t q = first[i]; q < first[i + 1]; q += kListGroup, g += 4) {
      g[0] = (int32_t)i;
      g[1] = q;
      g[2] = std::min<int32_t>(kListGroup, first[i + 1] - q);
      g[3] = 0;
    }
  for (int64_t k = 0; k < n_pairs; ++k) {
    const int32_t hk = hub(k), q = first[hk]++;
    a[q] = hk;
    b[q] = pi[k] == hk ? pj[k] : pi[k];
    pos[q] = (int32_t)k;
  }
}

}  // namespace

cudaError_t launch_pearson_list(VecStore &v, bool split, const int32_t *pi,
                                const int32_t *pj, int64_t n_pairs, double *out,
                                cudaStream_t s) {
  ListHost h;
  group_pairs(pi, pj, n_pairs, v.n, h);
  ListPlan L{};
  L.n_groups = h.n_groups;
  L.n_pairs = n_pairs;
  // slices that the touched rows share in L2, and enough of them to give every
  // SM sixteen warps; whole trips of 256 columns; fewer where the slices' sums
  // would take more than kListPartBytes
  constexpr int64_t kListPartBytes = 256ll << 20;
  const int64_t share = kListSliceBytes / (4 * h.n_rows);
  const int64_t spread = v.Dp * h.n_groups / (16 * (int64_t)num_sms());
  const int64_t most = std::max<int64_t>(kListPartBytes / (8 * n_pairs), 1);
  const int64_t least = (v.Dp + most - 1) / most;
  L.slice_cols = (std::max(std::max<int64_t>(std::min(share, spread), 1024), least) + 255) / 256 * 256;
  L.n_slices = (v.Dp + L.slice_cols - 1) / L.slice_cols;
  // the handle's list buffer (its lock held, and the call before has
  // synchronised its stream):
  // partial sums, then the index arrays
  const size_t head = (size_t)(L.n_slices * n_pairs) * sizeof(double);
  const size_t ints_at = (head + 15) / 16 * 16, bytes = ints_at + h.ints.size() * 4;
  cudaError_t e = cudaSuccess;
  if (v.list_bytes < bytes) {
    dfree(v.d_list);
    v.list_bytes = 0;
    e = dmalloc(&v.d_list, bytes + bytes / 4);
    if (e != cudaSuccess) return e;
    v.list_bytes = bytes + bytes / 4;
  }
  uint8_t *buf = v.d_list;
  // (a pageable source: staged before the call returns)
  e = cudaMemcpyAsync(buf + ints_at, h.ints.data(), h.ints.size() * 4, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    const int32_t *ints = reinterpret_cast<const int32_t *>(buf + ints_at);
    L.groups = reinterpret_cast<const int4 *>(ints);
    L.a = ints + 4 * h.n_groups;
    L.b = L.a + n_pairs;
    L.pos = L.b + n_pairs;
    double *part = reinterpret_cast<double *>(buf);
    const int64_t per_slice = (h.n_groups + kListThreads / 32 - 1) / (kListThreads / 32);
    const unsigned grid = (unsigned)std::min<int64_t>(per_slice * L.n_slices, 1 << 30);
    if (split)
      pearson_list_kernel<true><<<grid, kListThreads, 0, s>>>(v.d_hi, v.d_lo, nullptr, v.Dp, L,
                                                              part);
    else
      pearson_list_kernel<false><<<grid, kListThreads, 0, s>>>(nullptr, nullptr, v.d_c32, v.Dp, L,
                                                               part);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const unsigned g2 = (unsigned)std::min<int64_t>((n_pairs + 127) / 128, 65535);
    pearson_list_sum_kernel<<<g2, 128, 0, s>>>(part, L, v.d_rs, v.d_delta_all, v.D, out);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace ap

using namespace ap;

extern "C" ap_status ap_run_pairs_list(ap_items *it, int32_t fn, int32_t precision,
                                       const int32_t *pi, const int32_t *pj, int64_t n_pairs,
                                       const float *params, void *out, void *stream) {
  if (!it) return AP_ERR_INVALID_ARG;
  if (precision != AP_PREC_FP32 && precision != AP_PREC_SPLIT_BF16) return AP_ERR_INVALID_ARG;
  const bool cloud_fn = fn == AP_FN_OVERLAP || fn == AP_FN_GMM_L2 || fn == AP_FN_BHATTACHARYYA;
  const bool cloud = it->kind == AP_ITEMS_CLOUD2D || it->kind == AP_ITEMS_CLOUD3D;
  const bool ok_kind = cloud ? cloud_fn
                             : (it->kind == AP_ITEMS_VECTOR && fn == AP_FN_PEARSON) ||
                                   (it->kind == AP_ITEMS_SPARSE && fn == AP_FN_COSINE);
  if (!ok_kind) return AP_ERR_INVALID_ARG;
  if (params && it->kind != AP_ITEMS_CLOUD2D) return AP_ERR_INVALID_ARG;
  const int64_t n = cloud ? it->cl.n : it->kind == AP_ITEMS_SPARSE ? it->sp.n : it->vec.n;
  AP_TRY_ST(check_list(it, pi, pj, n_pairs, n));
  if (n_pairs == 0) return AP_OK;
  if (!out) return AP_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (!cloud) {
    const bool sparse = it->kind == AP_ITEMS_SPARSE;
    const bool split = precision == AP_PREC_SPLIT_BF16;
    if (!sparse) {
      const VecStore &v = it->vec;
      if (v.out_of_core) return AP_ERR_UNSUPPORTED;   // rows are not resident
      if ((split && !v.d_hi) || (!split && !v.d_c32)) return AP_ERR_STATE;
    }
    cudaError_t e = cudaSuccess;
    if (sparse) {
      int32_t *d_idx = nullptr;
      AP_TRY_ST(device_pairs(pi, pj, n_pairs, s, &d_idx));
      const SparseStore &sp = it->sp;
      const int grid = (int)std::min<int64_t>(n_pairs, (int64_t)num_sms() * 8);
      cosine_list_kernel<<<grid, kMergeThreads, 0, s>>>(sp.d_off, sp.d_idx, sp.d_val, sp.d_rs,
                                                         d_idx, d_idx + n_pairs, n_pairs,
                                                         reinterpret_cast<double *>(out));
      e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // before the index buffer goes
      dfree(d_idx);
    } else {
      // runs of several threads take the list buffer in turn
      std::lock_guard<std::mutex> lock(it->list_mutex);
      e = launch_pearson_list(it->vec, split, pi, pj, n_pairs, reinterpret_cast<double *>(out), s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    const ap_status st = e == cudaSuccess ? AP_OK : from_cuda(e);
    return st;
  }
  CloudStore lc;
  AP_TRY_ST(cloud_list_plan(it, pi, pj, n_pairs, s, lc));
  const int score = fn == AP_FN_GMM_L2 ? 1 : 2;
  if (fn != AP_FN_OVERLAP) AP_TRY_ST(ensure_score_storage(it, score, s));
  UnitQueue q;
  AP_TRY(take_queue(it, s, &q));
  if (fn == AP_FN_OVERLAP) {
    AP_TRY(launch_overlap(lc, params, reinterpret_cast<float *>(out), 0, q, s));
  } else {
    const CloudStore &c = it->cl;
    AP_TRY(launch_score(lc, score, c.d_pts_score[score - 1], c.d_lw_score[score - 1], c.d_self,
                        params, reinterpret_cast<float *>(out), q, s));
  }
  return AP_OK;
}

extern "C" ap_status ap_backward_list(ap_items *it, const int32_t *pi, const int32_t *pj,
                                      int64_t n_pairs, const float *params,
                                      const float *grad_out, float *grad_params, float *f_out,
                                      void *stream) {
  if (!it) return AP_ERR_INVALID_ARG;
  if (it->kind != AP_ITEMS_CLOUD2D) return AP_ERR_INVALID_ARG;
  AP_TRY_ST(check_list(it, pi, pj, n_pairs, it->cl.n));
  if (n_pairs == 0) return AP_OK;
  if (!grad_params) return AP_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  CloudStore lc;
  AP_TRY_ST(cloud_list_plan(it, pi, pj, n_pairs, s, lc));
  UnitQueue q;
  AP_TRY(take_queue(it, s, &q));
  AP_TRY(launch_overlap_grad_q(lc, q, params, grad_out, grad_params, f_out, 0.f, 0.f, nullptr,
                               nullptr, s));
  return AP_OK;
}

extern "C" ap_status ap_ascent_list(ap_items *it, const int32_t *pi, const int32_t *pj,
                                    int64_t n_pairs, float *params, int32_t n_steps, float eta,
                                    float fmin, float *f_out, int32_t *flags, void *stream) {
  if (!it) return AP_ERR_INVALID_ARG;
  if (it->kind != AP_ITEMS_CLOUD2D || n_steps < 0) return AP_ERR_INVALID_ARG;
  AP_TRY_ST(check_list(it, pi, pj, n_pairs, it->cl.n));
  if (n_pairs == 0 || n_steps == 0) return AP_OK;
  if (!params) return AP_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  CloudStore lc;
  AP_TRY_ST(cloud_list_plan(it, pi, pj, n_pairs, s, lc));
  for (int32_t k = 0; k < n_steps; ++k) {
    UnitQueue q;
    AP_TRY(take_queue(it, s, &q));
    AP_TRY(launch_overlap_grad_q(lc, q, nullptr, nullptr, nullptr, f_out, eta, fmin, params, flags,
                                 s));
  }
  return AP_OK;
}
