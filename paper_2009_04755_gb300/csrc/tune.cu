// tune.cu -- autotuner of the point-cloud tile plan, and CUDA-graph replay of
// the batched ascent (a run of one cost is one launch and needs no graph: the
// capture for each new output buffer cost a first pass 40 us).
//
// The tuner times every candidate plan (items per block, staged points per
// block, a-points per lane) on an evenly spread sample of its own tiles --
// about 2e10 point pairs, or everything when the workload is smaller -- and
// keeps the fastest.  The tile order stays the recursive quadrant order of
// the block grid (Sec. IV-B); what the tuner changes is the block size, i.e.
// how many items one tile reuses from shared memory and registers.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "ap_internal.h"

namespace ap {

int32_t min_reg_r(const CloudStore &c) {
  int64_t mx = 0;
  for (int64_t s : c.h_size) mx = std::max(mx, s);
  int32_t r = 2;                        // a-points go in pairs (FP32x2)
  while ((int64_t)r * 32 * kOverlapMaxRows < mx && r < 4) r *= 2;
  return r;
}

void clear_graphs(ap_items *it) {
  for (GraphEntry &g : it->graphs)
    if (g.exec) cudaGraphExecDestroy(g.exec);
  it->graphs.clear();
}

ap_status run_graphed(ap_items *it, const GraphKey &key, cudaStream_t s,
                      const std::function<cudaError_t(cudaStream_t)> &seq) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (s) AP_TRY(cudaStreamIsCapturing(s, &cap));
  if (cap != cudaStreamCaptureStatusNone) return from_cuda(seq(s));   // caller is capturing
  for (GraphEntry &g : it->graphs)
    if (g.key == key && g.plan_version == it->plan_version) return from_cuda(cudaGraphLaunch(g.exec, s));
  AP_TRY(cudaStreamBeginCapture(it->graph_stream, cudaStreamCaptureModeRelaxed));
  cudaError_t e = seq(it->graph_stream);
  cudaGraph_t graph = nullptr;
  cudaError_t e2 = cudaStreamEndCapture(it->graph_stream, &graph);
  if (e == cudaSuccess) e = e2;
  cudaGraphExec_t exec = nullptr;
  if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
  if (graph) cudaGraphDestroy(graph);
  if (e != cudaSuccess) return from_cuda(e);
  if (it->graphs.size() >= 16) {
    cudaGraphExecDestroy(it->graphs.front().exec);
    it->graphs.erase(it->graphs.begin());
  }
  it->graphs.push_back({key, it->plan_version, exec});
  return from_cuda(cudaGraphLaunch(exec, s));
}

namespace {

// point pairs of one block pair (I, J) of a candidate plan
double tile_cost(const std::vector<int32_t> &bstart, const std::vector<int64_t> &cnt, int32_t I,
                 int32_t J) {
  double si = 0, sj = 0, sq = 0;
  for (int32_t k = bstart[I]; k < bstart[I + 1]; ++k) { si += (double)cnt[k]; sq += (double)cnt[k] * cnt[k]; }
  if (I == J) return (si * si - sq) / 2;
  for (int32_t k = bstart[J]; k < bstart[J + 1]; ++k) sj += (double)cnt[k];
  return si * sj;
}

}  // namespace

// A set whose points fit many times into L2 gains nothing from the quadrant
// order's locality, but a queue of uneven tiles ends with a tail: such sets
// pop their tiles largest first (the greedy longest-first rule), so the last
// tiles taken are the small ones.
constexpr int64_t kLargestFirstBytes = 16ll << 20;

bool order_cloud_tiles(const std::vector<int32_t> &bstart, const std::vector<int64_t> &cnt,
                       int64_t total_pts, std::vector<int32_t> &tiles) {
  if (total_pts * (int64_t)(sizeof(float4) + sizeof(float)) > kLargestFirstBytes) return false;
  // counting sort on the cost in steps of a thousandth of the largest
  constexpr int kSteps = 1000;
  const size_t nt = tiles.size() / 2, nb = bstart.size() - 1;
  std::vector<double> sum(nb, 0.0), sq(nb, 0.0);
  for (size_t b = 0; b < nb; ++b)
    for (int32_t k = bstart[b]; k < bstart[b + 1]; ++k) {
      sum[b] += (double)cnt[k];
      sq[b] += (double)cnt[k] * (double)cnt[k];
    }
  std::vector<double> cost(nt);
  double most = 0.0;
  for (size_t t = 0; t < nt; ++t) {
    const int32_t I = tiles[2 * t], J = tiles[2 * t + 1];
    cost[t] = I == J ? (sum[I] * sum[I] - sq[I]) / 2 : sum[I] * sum[J];
    most = std::max(most, cost[t]);
  }
  std::vector<size_t> first(kSteps + 2, 0);
  auto step = [&](size_t t) {
    return most > 0.0 ? (size_t)((1.0 - cost[t] / most) * kSteps) : (size_t)0;
  };
  for (size_t t = 0; t < nt; ++t) ++first[step(t) + 1];
  for (size_t k = 1; k < first.size(); ++k) first[k] += first[k - 1];
  std::vector<int32_t> out(tiles.size());
  for (size_t t = 0; t < nt; ++t) {
    const size_t at = first[step(t)]++;
    out[2 * at] = tiles[2 * t];
    out[2 * at + 1] = tiles[2 * t + 1];
  }
  tiles.swap(out);
  return true;
}

}  // namespace ap

using namespace ap;

extern "C" ap_status ap_get_plan(const ap_items *it, ap_plan *out) {
  if (!it || !out) return AP_ERR_INVALID_ARG;
  out->k_split = 0;
  out->mma_ctas = 0;
  if (it->kind == AP_ITEMS_SPARSE) {
    out->block_items = out->block_pts = kSparseBlock;
    out->reg_r = out->sorted = 0;
    out->rate = 0.0;
    return AP_OK;
  }
  if (it->kind == AP_ITEMS_VECTOR) {
    out->block_items = kTcTileM;
    out->block_pts = kTcTileN;
    out->reg_r = 0;
    out->sorted = 0;
    out->rate = 0.0;
    out->k_split = it->vec.k_split;
    out->mma_ctas = it->vec.mma_ctas;
    return AP_OK;
  }
  out->block_items = it->cl.block_items;
  out->block_pts = it->cl.block_pts;
  out->reg_r = it->cl.reg_r;
  out->sorted = it->cl.sorted ? 1 : 0;
  out->rate = 0.0;
  return AP_OK;
}

namespace {
// whether the ranges of k_split keep to FP32 sums and their planes to the limit
bool planes_fit(int64_t k_split, int64_t Dp, int64_t pairs) {
  const int64_t nch = Dp / kOocChunkCols;
  return k_split > 0 && (nch + k_split - 1) / k_split * kOocChunkCols <= kKSplitCols &&
         k_split * pairs * (int64_t)sizeof(float) <= kPlaneBytes;
}
}  // namespace

// Column ranges per tile, in microseconds: a run costs ceil(units / slots)
// rounds of units, a unit its 64-column chunks (one each) and about kUnitUs
// more (the pipeline's start, and an epilogue that the next unit's MMAs cover
// for two chunks), and where its partial Grams go into planes the scaling pass
// one FP64 addition a pair and range.  Ranges of at most kKSplitCols columns,
// which the units in flight share in L2.  The cheapest wins.  1000 x 50,000, 10
// block pairs on 76 CTA pairs: 7 ranges fill one round and take 141 us with the
// scaling, 15 two rounds 167, 16 (the two units per SM of an earlier rule) a
// third round 206; 547 x 15,252, 6 block pairs: 12 ranges 50 us, 8 54, 16 68.
int32_t ap::default_k_split(int64_t n_tiles, int64_t slots, int64_t Dp, int64_t pairs) {
  constexpr double kUnitUs = 20.0, kPlaneAddsPerUs = 6e5;
  const int64_t nch = Dp / kOocChunkCols;
  const int64_t most = std::min<int64_t>(nch, kMaxKSplit);
  const int64_t least = std::min<int64_t>((Dp + kKSplitCols - 1) / kKSplitCols, most);
  int64_t best = least;
  double cost = 1e300;
  for (int64_t k = least; k <= most && n_tiles > 0; ++k) {
    const double rounds = (double)((n_tiles * k + slots - 1) / slots);
    const double unit = (double)((nch + k - 1) / k);
    const double c = rounds * (unit + kUnitUs) +
                     (pairs > 0 && planes_fit(k, Dp, pairs) ? (double)(k * pairs) / kPlaneAddsPerUs
                                                            : 0.0);
    if (c < cost) { cost = c; best = k; }
  }
  return best <= 1 ? 0 : (int32_t)best;
}

namespace {
ap_status upload_units(const std::vector<int32_t> &units, int32_t **d, int64_t *n) {
  dfree(*d);
  *n = 0;
  AP_TRY(dmalloc(d, std::max<size_t>(units.size(), kOocTileInts)));
  if (!units.empty())
    AP_TRY(upload_now(*d, units.data(), units.size() * 4));
  *n = (int64_t)units.size() / kOocTileInts;
  return AP_OK;
}
}  // namespace

// vector sets: (re)build the split-K wave units of the tensor-core tiles,
// for one CTA per tile (mma_ctas 1) or CTA pairs (mma_ctas 2; 0 = 2)
ap_status ap::set_vector_plan(ap_items *it, int32_t k_split, int32_t mma_ctas) {
  VecStore &v = it->vec;
  if (v.out_of_core) return AP_ERR_STATE;
  if (!v.d_hi) return AP_ERR_STATE;
  if (mma_ctas == 0) mma_ctas = 2;
  if (mma_ctas != 1 && mma_ctas != 2) return AP_ERR_INVALID_ARG;
  if (k_split < 0) {
    const int64_t nb = (v.n + kTcTileN - 1) / kTcTileN;
    k_split = mma_ctas == 2
                  ? default_k_split(nb * (nb + 1) / 2, tc2_pairs(), v.Dp, v.n * (v.n - 1) / 2)
                  : default_k_split(v.n_tiles_tc, num_sms(), v.Dp, 0);
  }
  cudaError_t e = cudaDeviceSynchronize();      // the old units may still be in use
  if (e != cudaSuccess) return from_cuda(e);
  dfree(v.d_panel_units);
  dfree(v.d_pair_units);
  dfree(v.d_pair_whole);
  dfree(v.d_planes);
  v.n_panel_units = v.n_pair_units = v.n_pair_whole = 0;
  v.k_split = 0;
  v.mma_ctas = mma_ctas;
  const int64_t nch = v.Dp / kOocChunkCols;
  std::vector<int32_t> units;
  if (mma_ctas == 2) {
    pair_units(v.n, nch, tc2_pairs(), 1, units);          // whole columns, one per macro pair
    AP_TRY_ST(upload_units(units, &v.d_pair_whole, &v.n_pair_whole));
  }
  if (k_split == 0) return AP_OK;
  if (mma_ctas == 2) {
    pair_units(v.n, nch, tc2_pairs(), k_split, units);
    AP_TRY_ST(upload_units(units, &v.d_pair_units, &v.n_pair_units));
    v.n_planes = std::min<int64_t>(k_split, nch);            // the ranges that were listed
    const int64_t P = v.n * (v.n - 1) / 2;
    if (P > 0 && planes_fit(v.n_planes, v.Dp, P) &&
        dmalloc(&v.d_planes, (size_t)(v.n_planes * P)) != cudaSuccess) {
      cudaGetLastError();                       // no room: the units add into the output
      v.d_planes = nullptr;
    }
  } else {
    panel_units(v.h_tiles_tc, nch, tc_grid(v.n_tiles_tc), k_split, units);
    AP_TRY_ST(upload_units(units, &v.d_panel_units, &v.n_panel_units));
  }
  v.k_split = k_split;
  return AP_OK;
}

extern "C" ap_status ap_set_plan(ap_items *it, const ap_plan *plan) {
  if (!it || !plan) return AP_ERR_INVALID_ARG;
  if (it->kind == AP_ITEMS_SPARSE) return AP_ERR_UNSUPPORTED;
  if (it->kind == AP_ITEMS_VECTOR) {
    if (plan->block_items != kTcTileM || plan->block_pts != kTcTileN) return AP_ERR_INVALID_ARG;
    if (plan->k_split < -1 || plan->k_split > kMaxKSplit) return AP_ERR_INVALID_ARG;
    if (plan->mma_ctas < 0 || plan->mma_ctas > 2) return AP_ERR_INVALID_ARG;
    return set_vector_plan(it, plan->k_split, plan->mma_ctas);
  }
  if (plan->block_items < 1 || plan->block_items > kOverlapMaxBlockItems) return AP_ERR_INVALID_ARG;
  if (plan->block_pts < 64 || plan->block_pts > 8192) return AP_ERR_INVALID_ARG;
  if (plan->reg_r != 2 && plan->reg_r != 4) return AP_ERR_INVALID_ARG;
  if (plan->reg_r < min_reg_r(it->cl)) return AP_ERR_INVALID_ARG;
  CloudPlanChoice ch{plan->block_items, plan->block_pts, plan->reg_r, it->cl.sorted};
  cudaError_t e = cudaDeviceSynchronize();      // the old plan may still be in use
  if (e != cudaSuccess) return from_cuda(e);
  AP_TRY_ST(build_cloud_plan(it, ch, nullptr));
  AP_TRY(cudaStreamSynchronize(nullptr));       // a run on any stream may follow
  return AP_OK;
}

extern "C" ap_status ap_tune(ap_items *it, int32_t mode, void *stream, ap_plan *out) {
  if (!it) return AP_ERR_INVALID_ARG;
  if (mode != 0 && mode != 1) return AP_ERR_INVALID_ARG;
  if (it->kind == AP_ITEMS_VECTOR || it->kind == AP_ITEMS_SPARSE) return AP_ERR_UNSUPPORTED;
  if (mode == 1 && it->kind != AP_ITEMS_CLOUD2D) return AP_ERR_INVALID_ARG;
  CloudStore &c = it->cl;
  if (c.n < 2) {
    if (out) ap_get_plan(it, out);
    return AP_OK;
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  std::vector<int64_t> cnt(c.n);
  for (int64_t k = 0; k < c.n; ++k) cnt[k] = c.h_size[c.h_perm[k]];
  const int64_t P = c.n * (c.n - 1) / 2;
  const double budget = 2e10;

  float *d_out = nullptr, *d_g = nullptr;
  CloudStore cand;                       // no plan buffers yet
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  ap_status st = AP_OK;
  cudaError_t e = dmalloc(&d_out, (size_t)P);
  if (e == cudaSuccess && mode == 1) e = dmalloc(&d_g, (size_t)P * 3);
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);

  CloudPlanChoice best{0, 0, 0, c.sorted};
  double best_rate = -1.0;
  const int32_t rmin = min_reg_r(c);
  for (int32_t rr : {2, 4}) {
    if (rr < rmin) continue;
    const int32_t bp = kCloudStagePts;           // more makes no other blocks
    for (int32_t bi : {2, 4, 8, 16, 32}) {
      if (e != cudaSuccess || st != AP_OK) break;
      CloudPlanHost plan;
      make_cloud_plan(c.h_poff, cnt, c.h_perm, 0, bi, bp, rr, plan);
      const std::vector<int32_t> &bstart = plan.bstart, &tiles = plan.tiles;
      const int64_t nt = (int64_t)tiles.size() / 2;
      std::vector<double> cost(nt);
      double total = 0;
      for (int64_t t = 0; t < nt; ++t) {
        cost[t] = tile_cost(bstart, cnt, tiles[2 * t], tiles[2 * t + 1]);
        total += cost[t];
      }
      // evenly spread sample of about `budget` point pairs, at least a few
      // tiles per SM
      int64_t stride = 1;
      if (total > budget) stride = (int64_t)std::ceil(total / budget);
      stride = std::min<int64_t>(stride, std::max<int64_t>(1, nt / (8LL * num_sms())));
      std::vector<int32_t> sample;
      double scost = 0;
      for (int64_t t = 0; t < nt; t += stride) {
        sample.push_back(tiles[2 * t]);
        sample.push_back(tiles[2 * t + 1]);
        scost += cost[t];
      }
      plan.tiles.swap(sample);
      // a shallow copy of the set with the sample's plan
      free_cloud_plan(cand);
      cand = c;
      cand.d_bmeta = cand.d_desc = cand.d_items = cand.d_tiles = nullptr;
      cand.block_items = bi;
      cand.block_pts = bp;
      cand.reg_r = rr;
      st = upload_cloud_plan(cand, plan, s);
      if (st != AP_OK) break;
      auto launch = [&]() {
        UnitQueue q;
        const cudaError_t taken = take_queue(it, s, &q);
        if (taken != cudaSuccess) return taken;
        return mode == 0 ? launch_overlap(cand, nullptr, d_out, 0, q, s)
                         : launch_overlap_grad_q(cand, q, nullptr, nullptr, d_g, d_out, 0.f, 0.f,
                                                 nullptr, nullptr, s);
      };
      float ms_best = 1e30f;
      e = launch();
      for (int rep = 0; rep < 2 && e == cudaSuccess; ++rep) {
        e = cudaEventRecord(e0, s);
        if (e == cudaSuccess) e = launch();
        if (e == cudaSuccess) e = cudaEventRecord(e1, s);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        float ms = 0;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        ms_best = std::min(ms_best, ms);
      }
      if (e != cudaSuccess) break;
      const double rate = scost / (ms_best * 1e-3);
      if (rate > best_rate) {
        best_rate = rate;
        best = {bi, bp, rr, c.sorted};
      }
    }
  }
  if (e != cudaSuccess) st = from_cuda(e);
  cudaStreamSynchronize(s);                      // the last candidate's plan is still in use
  dfree(d_out);
  dfree(d_g);
  free_cloud_plan(cand);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (st != AP_OK) return st;
  if (best_rate > 0) {
    st = build_cloud_plan(it, best, s);
    if (st != AP_OK) return st;
    AP_TRY(cudaStreamSynchronize(s));            // a run on any stream may follow
  }
  if (out) {
    ap_get_plan(it, out);
    out->rate = best_rate;
  }
  return AP_OK;
}
