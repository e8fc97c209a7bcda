// Host-side tile plan of the persistent products kernels: column tile widths of
// the two products, K slices of g_W, and which unit (CTA or CTA pair) takes
// which tiles in which order.
//
// A unit is a two-stage pipeline: its tensor-core stage works through the
// unit's tiles one after the other, its epilogue warps drain them in the same
// order, and two accumulator slots let tile i + 1 be multiplied while tile i is
// drained (tile i + 2 has to wait for tile i's slot).  The stages cost very
// different amounts per tile kind:
//   GX tile (g_x_hat^T = W^T g_y_hat^T, expanded by Eq. 7 in the epilogue): short
//           product (K = Cout), long epilogue (writes k*k / r times its size);
//   GW tile (g_W = g_y_hat^T x_hat): long product (K = all low-rank rows), short
//           epilogue.
// So a unit takes its GX tiles first and its GW tiles (or K slices of them)
// after: the GW products run under the GX epilogues, and the last thing a unit
// does is a short epilogue.  Tiles are handed out in one of two ways, whichever finishes
// first under the cost model below (measured on B200): greedily, each to the unit that
// would finish it first; or the GW tiles spread evenly and the GX tiles filled in around
// them, which is better where most units get both kinds (exact 768 -> 3072 with 8192
// tokens: greedily, the units without a GW tile idled at the end).  All tiles of a kind
// cost the same, so both ways are worked out by classes of units, and a candidate whose even
// share alone is longer than the best so far is not dealt at all: a first plan of 768 -> 3072
// with 512 blocks at rank 8 takes 0.2 ms of a host core instead of 5, exact 256 -> 256 with
// two million tokens 1 instead of 1500.
#include <cstdio>
#include <vector>

#include "lbp_fused.cuh"
#include "lbp_internal.h"

namespace lbp {

namespace {

// ---- cost model (microseconds) ----
// Operand delivery from L2 bounds the products: per SM about 95 GB/s to a GX tile, 76
// GB/s to a GW tile (all SMs at work: 11 TB/s).
constexpr double kFeedGxBytesPerUs = 95e3, kFeedGwBytesPerUs = 76e3;
constexpr double kTileFixedUs = 0.3;
// The expansion writes g_x at about 43 GB/s per SM (bound by the stores in flight, up
// to a 4 x 4 array, so channels past the edge cost nothing until the warps bind: 12
// blocks of 48 channels took 2.4 us in a tile of 128); with an 8 x 8 array the epilogue
// warps bind.  It takes four blocks at a time.
constexpr double kExpandBytesPerUs[3] = {43e3, 26e3, 18e3};
constexpr double kExpandWarpsBytesPerUs = 90e3;
constexpr double kGwStoreBytesPerUs = 45e3;
// K slices of g_W go through fp32 planes and one more kernel.
constexpr double kReduceFixedUs = 3.0;
constexpr double kReduceBytesPerUs = 4e6;

int ceil_div(int a, int b) { return (a + b - 1) / b; }

struct Costs {
  double mma_w, epi_w, mma_x, epi_x;
};

Costs tile_costs(const PlanShape& s, int bnw, int bnx, int bpt, int kbps) {
  const double a_bytes = 128.0 * 64 * 2;                       // a CTA's 128 rows of A per k-block
  const double bw = (s.pair ? bnw / 2 : bnw) * 64.0 * 2;       // its share of B
  const double bx = (s.pair ? bnx / 2 : bnx) * 64.0 * 2;
  Costs c;
  c.mma_w = kTileFixedUs + kbps * (a_bytes + bw) / kFeedGwBytesPerUs;
  c.mma_x = kTileFixedUs + s.num_kb_x * (a_bytes + bx) / kFeedGxBytesPerUs;
  c.epi_w = kTileFixedUs + 128.0 * bnw * 4 / kGwStoreBytesPerUs;
  if (s.epi_kind < 0) {
    c.epi_x = 0.5 + bnx * s.expand_bytes * 128.0 / kExpandBytesPerUs[0];
  } else {
    const double padded = (bpt + 3) / 4 * 4 * static_cast<double>(s.expand_bytes) * 128.0;
    const int row_tile = s.pair ? 256 : 128;
    const double used = static_cast<double>(s.gx_side) / (ceil_div(s.gx_side, row_tile) * row_tile);
    const double stores = padded * used / kExpandBytesPerUs[0];
    const double warps = padded / (s.epi_kind == 0 ? kExpandWarpsBytesPerUs : kExpandBytesPerUs[s.epi_kind]);
    c.epi_x = 0.5 + (stores > warps ? stores : warps);
  }
  return c;
}

// State of one unit while tiles are handed out.
struct Unit {
  double mma_free = 0, epi_free = 0;
  double slot_free[2] = {0, 0};   // when the epilogue has read the accumulator slot
  int n = 0;
  void take(double mma, double epi) {
    const double start = mma_free > slot_free[n & 1] ? mma_free : slot_free[n & 1];
    mma_free = start + mma;
    const double estart = mma_free > epi_free ? mma_free : epi_free;
    epi_free = estart + epi;
    slot_free[n & 1] = epi_free;   // the slot is read until (nearly) the end of the epilogue
    ++n;
  }
};

// Hands out n_gx GX tiles, then n_gw GW tiles greedily, each to the unit that would finish it
// first (the lowest numbered of several); returns the time the last unit finishes.  `owner`
// (optional) receives the unit of every tile, GX ids first.
//
// The units start alike and the tiles of a kind are alike, so the GX tiles go round the
// units, and from then on there are two classes of units, those that got one GX tile more
// and the others.  Within a class the next tile always goes to the next unit that has had
// the fewest, and which class it goes to changes only when all its units have had as many:
// the work is one step per tile of a unit, not one per tile and unit (a layer of 524288
// tokens took a second).
double deal_greedily(int units, int n_gx, int n_gw, const Costs& c, std::vector<int>* owner) {
  if (owner) {
    owner->assign(n_gx + n_gw, 0);
    for (int i = 0; i < n_gx; ++i) (*owner)[i] = i % units;
  }
  struct Class {
    int first, size;   // its units
    int dealt;         // how many of them have had a GW tile more than the others
    Unit now, next;    // the others, and those
    double finish;     // the next GW tile here
  } cls[2];
  cls[0].first = 0;
  cls[0].size = n_gx % units;
  cls[1].first = cls[0].size;
  cls[1].size = units - cls[0].size;
  Unit u;
  for (int i = 0; i < n_gx / units; ++i) u.take(c.mma_x, c.epi_x);
  cls[1].now = u;
  u.take(c.mma_x, c.epi_x);
  cls[0].now = u;
  auto look_ahead = [&](Class& k) {
    k.dealt = 0;
    k.next = k.now;
    k.next.take(c.mma_w, c.epi_w);
    k.finish = k.next.epi_free;
  };
  for (Class& k : cls) look_ahead(k);
  for (int i = 0; i < n_gw;) {
    Class& k = cls[0].size == 0 || cls[1].finish < cls[0].finish - 1e-9 ? cls[1] : cls[0];
    const int left = n_gw - i, n = k.size - k.dealt < left ? k.size - k.dealt : left;
    if (owner)
      for (int q = 0; q < n; ++q) (*owner)[n_gx + i + q] = k.first + k.dealt + q;
    i += n;
    k.dealt += n;
    if (k.dealt == k.size) {
      k.now = k.next;
      look_ahead(k);
    }
  }
  double last = 0;
  for (const Class& k : cls) {
    if (k.size == 0) continue;
    const double t = k.dealt > 0 ? k.next.epi_free : k.now.epi_free;
    last = t > last ? t : last;
  }
  return last;
}

// The GW tiles spread evenly: the last `more` units get one more of them than the others.
// Each of these two kinds of units gets as many GX tiles as lets the slower kind finish
// first.  Tiles are dealt in passes over the units, so that neighbouring tiles are worked
// on at the same time.
double deal_evenly(int units, int n_gx, int n_gw, const Costs& c, std::vector<int>* owner) {
  const int gw = n_gw / units, more = n_gw % units, less = units - more;
  std::vector<Unit> after_gx(1);   // a unit behind its first, second, ... GX tile
  auto unit_time = [&](int gx, int n) {
    while (static_cast<int>(after_gx.size()) <= gx) {
      after_gx.push_back(after_gx.back());
      after_gx.back().take(c.mma_x, c.epi_x);
    }
    Unit u = after_gx[gx];
    for (int i = 0; i < n; ++i) u.take(c.mma_w, c.epi_w);
    return u.epi_free;
  };
  auto gx_of_less = [&](int x) {   // GX tiles of the units with fewer GW tiles
    const long long rest = n_gx - static_cast<long long>(more) * x;
    const int y = rest <= 0 ? 0 : static_cast<int>((rest + less - 1) / less);
    return y == 0 && gw == 0 ? 1 : y;   // no unit without work
  };
  // Start where the units with fewer GW tiles could finish in the time that an even split of
  // the GX tiles takes (a unit needs at least the longer stage of each).
  int x0 = 0;
  if (more > 0) {
    const int x = n_gx / units;
    const double t0 = unit_time(x, gw + 1), t1 = unit_time(gx_of_less(x), gw), t = t0 > t1 ? t0 : t1;
    const long long y_most = static_cast<long long>(t / (c.mma_x > c.epi_x ? c.mma_x : c.epi_x)) + 1;
    const long long over = n_gx - y_most * less;
    if (over > 0) x0 = static_cast<int>((over + more - 1) / more);
  }
  double best = -1.0;
  int gx_more = 0, gx_less = 0;
  for (int x = x0; more == 0 ? x == 0 : x <= (n_gx + more - 1) / more; ++x) {
    const double t0 = more > 0 ? unit_time(x, gw + 1) : 0.0;
    if (best >= 0 && t0 > best) break;
    const int y = gx_of_less(x);
    const double t1 = unit_time(y, gw), t = t0 > t1 ? t0 : t1;
    if (best < 0 || t < best - 1e-9) {
      best = t;
      gx_more = x;
      gx_less = y;
    }
  }
  if (owner) {
    owner->assign(n_gx + n_gw, 0);
    for (int pass = 0, i = 0; i < n_gx; ++pass)
      for (int u = 0; u < units && i < n_gx; ++u)
        if (pass < (u < less ? gx_less : gx_more)) (*owner)[i++] = u;
    for (int pass = 0, i = 0; i < n_gw; ++pass)
      for (int u = 0; u < units && i < n_gw; ++u)
        if (pass < (u < less ? gw : gw + 1)) (*owner)[n_gx + i++] = u;
  }
  return best;
}

// Evenly only where that promises a clear gain: nearer than the model is accurate, the
// greedy order has the advantage that the units' lists differ in length.  (3 % is fitted, as
// the rates above are, to some dozen layers of 256 to 4096 channels: exact layers with as many
// GW tiles as units gain 14 % from the even deal, ties lose a few per cent.)
double deal(int units, int n_gx, int n_gw, const Costs& c, std::vector<int>* owner) {
  const double even = deal_evenly(units, n_gx, n_gw, c, nullptr);
  const double greedy = deal_greedily(units, n_gx, n_gw, c, nullptr);
  const bool evenly = even < 0.97 * greedy;
  if (owner != nullptr) {
    if (evenly)
      deal_evenly(units, n_gx, n_gw, c, owner);
    else
      deal_greedily(units, n_gx, n_gw, c, owner);
  }
  return evenly ? even : greedy;
}

bool same_shape(const PlanShape& a, const PlanShape& b) {
  return a.gw_rows == b.gw_rows && a.gw_cols == b.gw_cols && a.gx_side == b.gx_side &&
         a.blocks == b.blocks && a.piece == b.piece && a.n_extra == b.n_extra && a.units == b.units &&
         a.pair == b.pair && a.bnw_step == b.bnw_step && a.bnx_step == b.bnx_step &&
         a.bn_max == b.bn_max && a.max_splits == b.max_splits && a.expand_bytes == b.expand_bytes &&
         a.epi_kind == b.epi_kind && a.num_kb_w == b.num_kb_w && a.num_kb_x == b.num_kb_x;
}

// Tiles of this shape under given column tiles.
int count_gx(const PlanShape& s, int row_tile, int bnx, int bpt) {
  return ceil_div(s.gx_side, row_tile) * (ceil_div(s.blocks, bpt) + ceil_div(s.n_extra, bnx));
}
int count_gw(const PlanShape& s, int row_tile, int bnw, int splits) {
  return ceil_div(s.gw_rows, row_tile) * ceil_div(s.gw_cols, bnw) * splits;
}

struct Cached {
  PlanShape shape;
  TilePlan plan;
};

}  // namespace

const TilePlan& plan_products(const PlanShape& s) {
  static thread_local std::vector<Cached> cache;
  static thread_local size_t next = 0;
  for (const Cached& c : cache)
    if (same_shape(c.shape, s)) return c.plan;

  const int row_tile = s.pair ? 256 : 128;
  const int bnw_top = ceil_div(s.gw_cols, s.bnw_step) * s.bnw_step;   // no column tile wider than the matrix
  static const int kSplitChoices[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192};

  TilePlan best{};
  double best_t = -1.0;
  const TuneOptions& tune = tune_options();
  for (int bnw = s.bnw_step; bnw <= s.bn_max && bnw <= bnw_top; bnw += s.bnw_step) {
    for (int bnx = s.bnx_step; bnx <= s.bn_max; bnx += s.bnx_step) {
      if (bnx < s.piece) continue;
      // no wider than all pieces (or all single columns) together need
      const int less = bnx - s.bnx_step;
      if (less >= s.piece && less / s.piece >= s.blocks && less >= s.n_extra) continue;
      // Whole blocks that fit, or, in the narrowest tiles, fewer (what is left over is
      // multiplied and dropped): a few large blocks at a low rank would otherwise lie in a
      // handful of tiles (batch of 320 -> 1280 and 1280 -> 320, 36 blocks of 16 x 16 at rank
      // 1: 32 to a tile 88 us, up to 8 37 us).
      for (int bpt = bnx / s.piece; bpt > 0;
           bpt = bnx == 32 && count_gx(s, row_tile, bnx, bpt) < 2 * s.units ? bpt / 8 * 4 : 0) {
        for (int want : kSplitChoices) {
          if (want > 1 && (want > s.max_splits || want > s.num_kb_w / 4)) continue;
          if (tune.has_tiles &&
              (bnw != tune.tiles_bnw || bnx != tune.tiles_bnx || want != tune.tiles_splits))
            continue;
          const int kbps = ceil_div(s.num_kb_w, want);
          const int splits = ceil_div(s.num_kb_w, kbps);
          const int n_gw = count_gw(s, row_tile, bnw, splits), n_gx = count_gx(s, row_tile, bnx, bpt);
          const Costs c = tile_costs(s, bnw, bnx, bpt, kbps);
          const int units = n_gw + n_gx < s.units ? n_gw + n_gx : s.units;
          const double reduce =
              splits > 1 ? kReduceFixedUs +
                               (splits + 1.0) * s.gw_rows * static_cast<double>(s.gw_cols) * 4 / kReduceBytesPerUs
                         : 0.0;
          // an even share of either stage is the least it can take: most candidates end here
          const double mma = n_gx * c.mma_x + n_gw * c.mma_w, epi = n_gx * c.epi_x + n_gw * c.epi_w;
          if (best_t >= 0 && (mma > epi ? mma : epi) / units + reduce >= best_t) continue;
          const double t = deal(units, n_gx, n_gw, c, nullptr) + reduce;
          if (best_t < 0 || t < best_t - 1e-9) {
            best_t = t;
            best.BNw = bnw;
            best.BNx = bnx;
            best.bpt = bpt;
            best.splits = splits;
            best.kbps = kbps;
          }
        }
      }
    }
  }
  best.model_us = best_t;
  if (best_t < 0) {   // an override that fits nothing: the widest tiles, no slices
    best.BNw = bnw_top < s.bn_max ? bnw_top : s.bn_max;
    best.BNx = s.bn_max;
    best.bpt = s.bn_max / s.piece;
    best.splits = 1;
    best.kbps = s.num_kb_w;
  }

  // per-unit tile lists of the chosen plan
  const int n_gw = count_gw(s, row_tile, best.BNw, best.splits);
  const int n_gx = count_gx(s, row_tile, best.BNx, best.bpt);
  const int units = n_gw + n_gx < s.units ? n_gw + n_gx : s.units;
  FusedSchedule& sc = best.sched;
  sc.listed = 0;
  if (n_gw + n_gx <= kSchedMaxItems && units <= kSchedMaxUnits) {
    std::vector<int> owner;
    deal(units, n_gx, n_gw, tile_costs(s, best.BNw, best.BNx, best.bpt, best.kbps), &owner);
    std::vector<std::vector<uint16_t>> lists(units);
    // tile ids as the kernels number them: the GW tiles come first
    for (int i = 0; i < n_gx; ++i) lists[owner[i]].push_back(static_cast<uint16_t>(n_gw + i));
    for (int i = 0; i < n_gw; ++i) lists[owner[n_gx + i]].push_back(static_cast<uint16_t>(i));
    int at = 0;
    for (int uidx = 0; uidx < units; ++uidx) {
      sc.first[uidx] = static_cast<uint16_t>(at);
      for (uint16_t id : lists[uidx]) sc.ids[at++] = id;
    }
    for (int uidx = units; uidx <= kSchedMaxUnits; ++uidx) sc.first[uidx] = static_cast<uint16_t>(at);
    sc.listed = 1;
  }
  if (tune.verbose)
    fprintf(stderr, "lbp products plan (%s): BNw=%d BNx=%d (%d blocks) gw_splits=%d kb/split=%d tiles=%d+%d "
                    "units=%d listed=%d model=%.1f us\n",
            s.pair ? "CTA pairs" : "CTAs", best.BNw, best.BNx, best.bpt, best.splits, best.kbps, n_gx, n_gw,
            units, sc.listed, best_t);

  if (cache.capacity() < 128) cache.reserve(128);
  if (cache.size() < 128) {
    cache.push_back(Cached{s, best});
    return cache.back().plan;
  }
  cache[next] = Cached{s, best};
  const TilePlan& out = cache[next].plan;
  next = (next + 1) % cache.size();
  return out;
}

}  // namespace lbp
