// plan.cpp -- host-side schedule of the all-pairs library.
//
// The upper triangle of the item grid is walked in recursively blocked tiles
// (Sec. IV-B: the matrix is split into four quadrants, each quadrant again,
// quadrants without work are skipped).  Here the recursion stops at blocks of
// items; the resulting list of block pairs (I <= J) is what the persistent
// kernels pop from their atomic queue, so consecutive tiles share item blocks
// and stay warm in L2 and shared memory.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "ap_internal.h"

namespace ap {

namespace {
struct Region { int64_t r0, r1, c0, c1; };
}

void dc_block_pairs(int64_t nb, std::vector<int32_t> &out) {
  out.clear();
  if (nb <= 0) return;
  // explicit stack; children pushed in reverse so they pop as TL, TR, BL, BR
  std::vector<Region> stack;
  stack.push_back({0, nb, 0, nb});
  while (!stack.empty()) {
    Region g = stack.back();
    stack.pop_back();
    if (g.r0 >= g.r1 || g.c0 >= g.c1) continue;
    if (g.r0 > g.c1 - 1) continue;            // every block below the diagonal
    if (g.r1 - g.r0 == 1 && g.c1 - g.c0 == 1) {
      out.push_back((int32_t)g.r0);           // block pair (I, J), I <= J
      out.push_back((int32_t)g.c0);
      continue;
    }
    int64_t rm = g.r0 + (g.r1 - g.r0 + 1) / 2;
    int64_t cm = g.c0 + (g.c1 - g.c0 + 1) / 2;
    stack.push_back({rm, g.r1, cm, g.c1});    // bottom-right (visited last)
    stack.push_back({rm, g.r1, g.c0, cm});    // bottom-left
    stack.push_back({g.r0, rm, cm, g.c1});    // top-right
    stack.push_back({g.r0, rm, g.c0, cm});    // top-left (visited first)
  }
}

void make_blocks(const std::vector<int64_t> &poff, const std::vector<int64_t> &cnt,
                 int32_t max_items, int64_t max_pts, int32_t reg_r, int64_t max_rows,
                 std::vector<int32_t> &bstart) {
  bstart.clear();
  int64_t n = (int64_t)poff.size() - 1;
  int64_t i = 0;
  while (i < n) {
    bstart.push_back((int32_t)i);
    int64_t pts = 0, k = 0, rows = 0;
    while (i < n && k < max_items) {
      int64_t sz = poff[i + 1] - poff[i];
      int64_t r = cloud_rows(cnt[i], reg_r);
      if (k > 0 && (pts + sz > max_pts || rows + r > max_rows)) break;
      pts += sz;
      rows += r;
      ++k;
      ++i;
    }
  }
  bstart.push_back((int32_t)n);
}

namespace {
// a piece of an item: `groups` (1..8) groups from `grp`
struct Piece { int32_t grp, groups, row, il; };
// eight groups' worth of lanes, holding pieces in a row
struct Slot {
  int32_t n, room;
  Piece p[8];
};

// one job of up to R slots
void emit_job(const Slot *slots, int32_t count, std::vector<int32_t> &desc) {
  const int32_t re = job_re(count), lpg = 4 >> re;
  const size_t at = desc.size();
  desc.resize(at + 64);
  int32_t *d = desc.data() + at;
  for (int l = 0; l < 32; ++l) {
    d[2 * l] = -1;
    d[2 * l + 1] = pack_lane(0, 0, 1, 0, re, 0);
  }
  for (int32_t s = 0; s < count; ++s) {
    int32_t go = 0;                              // groups of the slot in use
    for (int32_t k = 0; k < slots[s].n; ++k) {
      const Piece &p = slots[s].p[k];
      for (int32_t q = 0; q < p.groups * lpg; ++q) {
        const int32_t lane = (s * 8 + go) * lpg + q;
        d[2 * lane] = p.grp + q / lpg;
        d[2 * lane + 1] = pack_lane(p.row, q, p.groups * lpg, p.il, re, q % lpg);
      }
      go += p.groups;
    }
  }
}

// the jobs of a block of several items
void pack_block(const std::vector<int64_t> &poff, const std::vector<int64_t> &cnt, int32_t i0,
                int32_t i1, int32_t reg_r, std::vector<Slot> &slots,
                std::vector<Piece> &part, std::vector<int32_t> &desc) {
  slots.clear();
  part.clear();
  int32_t rows = 0;
  for (int32_t i = i0; i < i1; ++i) {
    const int32_t grp0 = (int32_t)(poff[i] / 4), G = (int32_t)((cnt[i] + 3) / 4);
    const int32_t full = 8 * reg_r, nfull = G / full;
    for (int32_t k = 0; k < nfull; ++k)
      for (int32_t lane = 0; lane < 32; ++lane) {
        const int2 d = cloud_lane_desc(k, lane, grp0, G, reg_r, rows, i - i0);
        desc.push_back(d.x);
        desc.push_back(d.y);
      }
    for (int32_t g = nfull * full, r = rows + nfull; g < G; g += 8, ++r) {
      const Piece p{grp0 + g, std::min(8, G - g), r, i - i0};
      if (p.groups == 8) slots.push_back({1, 0, {p}});
      else part.push_back(p);
    }
    rows += cloud_rows(cnt[i], reg_r);
  }
  // pieces of fewer than 8 groups share slots: largest first, first fit
  std::stable_sort(part.begin(), part.end(),
                   [](const Piece &a, const Piece &c) { return a.groups > c.groups; });
  const size_t first = slots.size();
  for (const Piece &p : part) {
    size_t s = first;
    while (s < slots.size() && slots[s].room < p.groups) ++s;
    if (s == slots.size()) slots.push_back({0, 8, {}});
    slots[s].p[slots[s].n++] = p;
    slots[s].room -= p.groups;
  }
  for (size_t s = 0; s < slots.size(); s += reg_r)
    emit_job(&slots[s], (int32_t)std::min<size_t>(slots.size() - s, reg_r), desc);
}
}  // namespace

void make_cloud_plan(const std::vector<int64_t> &poff, const std::vector<int64_t> &cnt,
                     const std::vector<int32_t> &perm, int64_t split_tail, int32_t block_items,
                     int32_t block_pts, int32_t reg_r, CloudPlanHost &out) {
  out = CloudPlanHost();
  // several items fit the staging buffer: a window that cut one of them would
  // sum it in another order than other plans do, and lose its boxes
  make_blocks(poff, cnt, block_items, std::min(block_pts, kCloudStagePts), reg_r,
              kOverlapMaxRows, out.bstart);
  const int64_t nb = (int64_t)out.bstart.size() - 1, n = (int64_t)cnt.size();
  out.items.resize((size_t)n * 4);
  out.bmeta.reserve((size_t)(nb + n) * 8);
  std::vector<Slot> slots;
  std::vector<Piece> part;
  for (int64_t b = 0; b < nb; ++b) {
    const int32_t i0 = out.bstart[b], i1 = out.bstart[b + 1];
    int32_t rows = 0, job0 = -1, jobs = 0;
    for (int32_t i = i0; i < i1; ++i) {
      int32_t *m = &out.items[4 * (size_t)i];
      m[0] = (int32_t)(poff[i] / 4);
      m[1] = (int32_t)cnt[i];
      m[2] = perm[i];
      m[3] = rows;
      rows += cloud_rows(cnt[i], reg_r);
    }
    if (i1 - i0 == 1) {
      jobs = (int32_t)(((cnt[i0] + 3) / 4 + 8 * reg_r - 1) / (8 * reg_r));
    } else {
      job0 = (int32_t)(out.desc.size() / 64);
      pack_block(poff, cnt, i0, i1, reg_r, slots, part, out.desc);
      jobs = (int32_t)(out.desc.size() / 64) - job0;
    }
    const int32_t pts = (int32_t)(poff[i1] - poff[i0]);
    const int32_t m[8] = {i0, i1, (int32_t)(poff[i0] / 4), pts / 4, job0, jobs, rows, 0};
    out.bmeta.insert(out.bmeta.end(), m, m + 8);
    out.max_rows = std::max(out.max_rows, rows);
    out.max_items = std::max(out.max_items, i1 - i0);
    out.max_pts = std::max(out.max_pts, pts);
  }
  dc_block_pairs(nb, out.tiles);
  out.largest_first = order_cloud_tiles(out.bstart, cnt, poff[n], out.tiles);
  // the tail: one tile per item of J, so that the CTAs run dry together
  const size_t nt = out.tiles.size() / 2;
  const size_t keep = nt > (size_t)split_tail ? nt - (size_t)split_tail : 0;
  std::vector<int32_t> tail, single((size_t)n, -1);
  for (size_t t = keep; t < nt; ++t) {
    const int32_t I = out.tiles[2 * t], J = out.tiles[2 * t + 1];
    const int32_t j0 = out.bstart[J], j1 = out.bstart[J + 1];
    for (int32_t j = j0; j < j1; ++j) {
      if (I == J && j == j0) continue;           // no i < j
      int32_t b = J;
      if (j1 - j0 > 1) {
        if (single[j] < 0) {
          single[j] = (int32_t)(out.bmeta.size() / 8);
          const int32_t m[8] = {j, j + 1, (int32_t)(poff[j] / 4),
                                (int32_t)((poff[j + 1] - poff[j]) / 4), -1, 0, 0, 0};
          out.bmeta.insert(out.bmeta.end(), m, m + 8);
        }
        b = single[j];
      }
      tail.push_back(I);
      tail.push_back(b);
    }
  }
  out.tiles.resize(2 * keep);
  out.tiles.insert(out.tiles.end(), tail.begin(), tail.end());
}

void single_item_blocks(const CloudStore &c, int32_t reg_r, std::vector<int32_t> &bmeta) {
  bmeta.clear();
  for (int64_t i = 0; i < c.n; ++i) {
    const int64_t cnt = c.h_size[c.h_perm[i]], G = (cnt + 3) / 4, full = 8 * reg_r;
    const int32_t m[8] = {(int32_t)i, (int32_t)i + 1, (int32_t)(c.h_poff[i] / 4), (int32_t)G, -1,
                          (int32_t)((G + full - 1) / full), cloud_rows(cnt, reg_r), 0};
    bmeta.insert(bmeta.end(), m, m + 8);
  }
}

void tc_tiles(int64_t n, std::vector<int32_t> &tiles) {
  // macro grid of kTcTileN items; each macro pair (I <= J) holds two row
  // halves of kTcTileM items, kept when they contain some pair i < j.
  tiles.clear();
  int64_t nb = (n + kTcTileN - 1) / kTcTileN;
  std::vector<int32_t> macro;
  dc_block_pairs(nb, macro);
  const int64_t halves = kTcTileN / kTcTileM;
  for (size_t t = 0; t < macro.size(); t += 2) {
    int64_t I = macro[t], J = macro[t + 1];
    for (int64_t h = 0; h < halves; ++h) {
      int64_t ib = I * halves + h;
      int64_t i0 = ib * kTcTileM;
      int64_t jmax = std::min<int64_t>(J * kTcTileN + kTcTileN, n) - 1;
      if (i0 >= n || i0 >= jmax) continue;   // no i < j in this half
      tiles.push_back((int32_t)ib);
      tiles.push_back((int32_t)J);
    }
  }
}

void panel_units(const std::vector<int32_t> &tiles, int64_t nchunks, int64_t group,
                 int64_t k_split, std::vector<int32_t> &units) {
  // waves of `group` consecutive tiles; inside a wave, column range p of
  // every tile before range p + 1 of any, so the tiles running at one time
  // stream the same columns of their rows
  units.clear();
  const int64_t nt = (int64_t)tiles.size() / 2;
  k_split = std::max<int64_t>(1, std::min<int64_t>(k_split, nchunks));
  for (int64_t w0 = 0; w0 < nt; w0 += group) {
    const int64_t w1 = std::min<int64_t>(nt, w0 + group);
    for (int64_t p = 0; p < k_split; ++p) {
      const int32_t c0 = (int32_t)(p * nchunks / k_split);
      const int32_t c1 = (int32_t)((p + 1) * nchunks / k_split);
      for (int64_t t = w0; t < w1; ++t) {
        const int32_t ib = tiles[2 * t], jb = tiles[2 * t + 1];
        const int32_t rb = jb * (kTcTileN / kTcTileM);
        const int32_t u[kOocTileInts] = {ib, rb, rb + 1, ib, jb, c0, c1, 0};
        units.insert(units.end(), u, u + kOocTileInts);
      }
    }
  }
}

void pair_units(int64_t n, int64_t nchunks, int64_t group, int64_t k_split,
                std::vector<int32_t> &units) {
  std::vector<int32_t> macro;
  dc_block_pairs((n + kTcTileN - 1) / kTcTileN, macro);
  pair_units_of(macro, nchunks, group, k_split, units);
}

void pair_units_of(const std::vector<int32_t> &macro, int64_t nchunks, int64_t group,
                   int64_t k_split, std::vector<int32_t> &units) {
  // macro pairs of 256 items; each CTA of a pair takes one 128-item half of
  // the I macro and stages one half of the J macro
  units.clear();
  const int64_t nt = (int64_t)macro.size() / 2;
  k_split = std::max<int64_t>(1, std::min<int64_t>(k_split, nchunks));
  group = std::max<int64_t>(1, group);
  for (int64_t w0 = 0; w0 < nt; w0 += group) {
    const int64_t w1 = std::min<int64_t>(nt, w0 + group);
    for (int64_t p = 0; p < k_split; ++p) {
      const int32_t c0 = (int32_t)(p * nchunks / k_split);
      const int32_t c1 = (int32_t)((p + 1) * nchunks / k_split);
      for (int64_t t = w0; t < w1; ++t) {
        const int32_t I = macro[2 * t], J = macro[2 * t + 1];
        const int32_t u[kOocTileInts] = {2 * I, 2 * I + 1, 2 * J, 2 * J + 1, 2 * I, J, c0, c1};
        units.insert(units.end(), u, u + kOocTileInts);
      }
    }
  }
}

}  // namespace ap
