// Declarations of the persistent products + expansion kernel (bf16 data).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "lbp_internal.h"

namespace lbp {

// Highest rank the persistent products kernel takes: the tensor-pipe projection must
// produce that many rows per block (orders 8 and 16: up to 48, which covers LP_L1-6,
// LP_L1-7 and LP_L1-8 of the paper's tables; order 4: all 16).
inline int fused_max_rank(int k) { return k == 4 ? 16 : 48; }

// Scaling inside the products path.  Eq. 6-7 put 1/k on either side of the
// products; all of it is powers of two, so it can sit anywhere without changing
// a bit of the results.  Here g_y_hat carries 1/k^2 and x_hat none: g_W =
// g_y_hat^T x_hat comes out right, and g_x_hat = g_y_hat W already holds the 1/k
// of the reverse projection, which then only adds, subtracts and rounds.  Where
// x_hat was taken at forward time (orthonormal coefficients) g_y_hat carries 1/k
// too and the expansion multiplies by the other 1/k.
inline float fused_scale_gy(int k, bool x_hat_given) {
  return 1.0f / static_cast<float>(x_hat_given ? k : k * k);
}
inline float fused_scale_x(int) { return 1.0f; }

struct FusedParams {
  // token grid and low-rank rows: block blk owns rows blk * r .. blk * r + r - 1 of
  // x_hat / g_y_hat (dense); nb = 0: no grid, only tokens that take Eq. 2
  int32_t nb, Hb, Wb, H, W, r;
  int32_t Cin, Cout;
  // GX: tiles of 128 channels per CTA x BNx low-rank rows; a tile's rows are those of
  // bpt whole blocks (what BNx leaves over is multiplied and dropped)
  int32_t BNx, bpt, n_ct, n_rt, num_kb_x;   // channel tiles, row tiles, k-blocks (Cout / 64)
  // GW: 128 rows of g_W per CTA x BNw columns; k-blocks of the low-rank rows, then of
  // the tokens outside the grid
  int32_t BNw, mt_w, nt_w, kb_lr, num_kb_w;
  int32_t n_gx_tiles, n_gw_tiles;         // n_gw_tiles counts K slices: mt_w * nt_w * gw_splits
  int32_t gw_splits, kb_per_split_w;      // K slices of a GW tile (fp32 planes, reduced afterwards)
  float* gw_planes;                       // [gw_splits][Cout][Cin] when gw_splits > 1
  int32_t gw_bf16;
  float beta;                             // g_W <- beta * g_W + ... (0: overwritten, not read)
  float gx_scale;                         // factor of g_x_hat ahead of the expansion (a power of two)
  int32_t n_extra;                        // tokens outside the grid (Eq. 2): GX tiles behind the grid's
  void* g_W;
  uint32_t* status;
  // failure-injection hook of the test suite (lbp_test_stall_products): the TMA
  // producers issue no load, so every other role runs into its bounded wait
  int32_t test_stall;
#ifdef LBP_ROLE_TRACE
  unsigned long long* trace;              // role timeline, kTraceSlots slots per CTA (null = off)
#endif
};

// Which unit (a CTA, or a CTA pair) works on which tiles, in which order: planned
// on the host (lbp_fused_plan.cu) and handed to the kernel as a launch
// parameter.  Tile ids: [0, n_gw_tiles) are the GW tiles (id = tile * gw_splits +
// K slice), then the GX tiles (row tile, channel tile).
constexpr int kSchedMaxItems = 1536;
constexpr int kSchedMaxUnits = 160;
struct FusedSchedule {
  int32_t listed;                        // 0: too many tiles for the table, the units deal them by formula
  uint16_t first[kSchedMaxUnits + 1];    // tiles of unit u: ids[first[u]] .. ids[first[u + 1] - 1]
  uint16_t ids[kSchedMaxItems];
};

// One tile of work as the kernel sees it.
struct WorkTile {
  int is_gw;
  int a, b;        // GW: (row tile i, column tile j) ; GX: (row tile m, channel tile n); m >= n_rt: extra tokens
  int kb0, n_kb;   // k-block range (a K slice for GW)
  int slice;
};

#ifdef __CUDACC__
__device__ __forceinline__ int unit_tile_count(const FusedParams& p, const FusedSchedule& sc, int unit,
                                               int units);
__device__ __forceinline__ WorkTile unit_tile(const FusedParams& p, const FusedSchedule& sc, int unit,
                                              int units, int nth);
#endif

// How the expansion finds a block's coefficients: natural-order LB x LB position ->
// accumulator column inside the block's columns, and what to AND the value with
// (all ones, or zero where the basis is not selected; col is 0 there).  Forms with
// an 8 x 8 array keep it as four 4 x 4 quadrants (see Expand).
struct FusedBasis {
  int32_t col[64];
  uint32_t keep[64];
  // 1: the slots of a block are ordered by rows (i, then j) and every row holds j = 0 ..
  // n_i - 1 only: row i starts at column row[i] and is read with one wide load
  int32_t by_rows;
  int32_t row[8];
  // sparse form: the one basis with i >= 4 (side 0) and the one with j >= 4 (side 1)
  int32_t ex_col[2];
  uint32_t ex_keep[2];
  float ex_sign[2][16];      // +-1: sign of that basis on the 4 x 4 patches
};

// Builds with -DLBP_ROLE_TRACE carry a per-CTA role timeline (diagnostics) in
// the last bytes of the scratch region; ordinary builds have neither the code
// nor the bytes.
#ifdef LBP_ROLE_TRACE
constexpr int kTraceSlots = 128;   // 8-byte slots per CTA: 8 for the roles, then 8 per tile
constexpr size_t kFusedTraceBytes = 256 * kTraceSlots * 8;
#else
constexpr size_t kFusedTraceBytes = 0;
#endif

struct FusedLayout {
  size_t x_hat, gy_hat, planes, planes_bytes, trace, total;
};

// Side-stream mode of one call (set per thread by lbp_backward_batch): the
// projection goes to `proj_stream` on at most `proj_ctas` CTAs (0 = all SMs),
// `proj_done` is recorded behind it and the products kernel, on `prod_units`
// CTA pairs (0 = all), waits for it on the call's own stream.
struct FusedOverlap {
  cudaStream_t proj_stream;
  cudaEvent_t proj_done;
  int proj_ctas;
  int prod_units;
};
void set_fused_overlap(const FusedOverlap* ov);   // nullptr = off
const FusedOverlap* fused_overlap();

// Per-thread switch set by lbp_test_stall_products (test hook).
void set_test_stall(bool on);
bool test_stall();
void set_test_stall_projection(bool on);
bool test_stall_projection();

#ifdef __CUDACC__
// Without a table the tiles are dealt in a snake over the units (first pass
// forwards, second backwards, ...), in id order.
__device__ __forceinline__ int unit_tile_count(const FusedParams& p, const FusedSchedule& sc, int unit,
                                               int units) {
  if (sc.listed) return static_cast<int>(sc.first[unit + 1]) - static_cast<int>(sc.first[unit]);
  const int total = p.n_gw_tiles + p.n_gx_tiles;
  int n = 0;
  for (int round = 0; round * units < total; ++round) {
    const int pos = (round & 1) ? (units - 1 - unit) : unit;
    if (round * units + pos < total) ++n;
  }
  return n;
}
__device__ __forceinline__ WorkTile unit_tile(const FusedParams& p, const FusedSchedule& sc, int unit,
                                              int units, int nth) {
  int id = 0;
  if (sc.listed) {
    id = sc.ids[sc.first[unit] + nth];
  } else {
    // every pass of the snake gives a unit one tile, the last one perhaps none
    const int pos = (nth & 1) ? (units - 1 - unit) : unit;
    id = nth * units + pos;
  }
  WorkTile tl;
  if (id < p.n_gw_tiles) {
    tl.is_gw = 1;
    const int t = id / p.gw_splits;
    tl.slice = id - t * p.gw_splits;
    tl.a = t / p.nt_w;
    tl.b = t - tl.a * p.nt_w;
    tl.kb0 = tl.slice * p.kb_per_split_w;
    const int end = tl.kb0 + p.kb_per_split_w;
    tl.n_kb = (end < p.num_kb_w ? end : p.num_kb_w) - tl.kb0;
  } else {
    id -= p.n_gw_tiles;
    tl.is_gw = 0;
    tl.slice = 0;
    tl.a = id / p.n_ct;
    tl.b = id - tl.a * p.n_ct;
    tl.kb0 = 0;
    tl.n_kb = p.num_kb_x;
  }
  return tl;
}
#endif

// ---- host-side tile plan (lbp_fused_plan.cu) ----
// GW tiles: row_tile x BNw pieces of a gw_rows x gw_cols matrix, num_kb_w k-blocks
// deep, possibly in K slices.  GX tiles: row_tile of the fixed side (gx_side) x BNx of
// the other, num_kb_x k-blocks deep; the other side is made of `blocks` indivisible
// pieces of `piece` columns, plus `n_extra` single columns in tiles of their own.  A
// unit is a CTA (row_tile 128) or a CTA pair (256).
struct PlanShape {
  int gw_rows, gw_cols;
  int gx_side;
  int blocks, piece, n_extra;
  int units, pair;
  int bnw_step, bnx_step, bn_max;   // column tiles: multiples of the step up to bn_max
  int max_splits;                   // K slices of g_W the scratch has planes for
  int expand_bytes;                 // what the epilogue of a GX tile writes per piece and channel
  int epi_kind;                     // expansion: 0 up to a 4 x 4 array, 1 sparse 8 x 8, 2 8 x 8; -1 none
  int num_kb_w, num_kb_x;
};
struct TilePlan {
  int BNw, BNx, splits, kbps;
  int bpt;           // blocks of a GX tile
  double model_us;   // time of the products kernel under the planner's cost model
  FusedSchedule sched;
};
// Column tiles, K slices of g_W and the per-unit tile lists for this shape
// (remembered per calling thread for recent shapes).
const TilePlan& plan_products(const PlanShape& s);

// Called between the projection launch and the products launch (phase events).
using FusedPhaseHook = int (*)(void* arg, cudaStream_t stream);

bool fused_supported(const lbp_layer& L, const BasisPlan& bp);
size_t fused_scratch_bytes(const lbp_layer& L, int r, FusedLayout* lay);
// Strides of the three token tensors of a call (an entry that is all zero: dense).
struct CallViews {
  lbp_view x, gy, gx;
};
// What lbp_extras adds to the products kernel: accumulation into g_W and the
// tokens outside the grid (pitches in elements, 0: dense).
struct FusedExtras {
  float beta;
  int n_extra;
  const void* x;
  const void* gy;
  void* gx;
  long long x_pitch, gy_pitch, gx_pitch;
};
// Exactly one of x / x_hat_dense is given; x_hat_dense are coefficients p(x)
// taken earlier, stored densely (blocks * r, Cin).  views: null = all dense.
// dc_slot: receives the slot of basis (0, 0) in g_y_hat, -1 = not selected.
int launch_fused(const void* x, const void* x_hat_dense, const void* g_y, const void* W, void* g_x,
                 void* g_W, const lbp_layer& L, const BasisPlan& bp, uint8_t* scratch,
                 uint32_t* status, cudaStream_t stream, FusedPhaseHook hook, void* hook_arg,
                 const CallViews* views = nullptr, const FusedExtras* extras = nullptr,
                 int* dc_slot = nullptr);

// Eq. 2 (exact backpropagation, bf16) over `tokens` dense tokens: both products in one
// launch of the products kernel, every token outside the grid.  planes: scratch for K
// slices of g_W.
int launch_exact(const void* x, const void* g_y, const void* W, void* g_x, void* g_W, const lbp_layer& L,
                 long long tokens, float* planes, size_t planes_bytes, uint32_t* status, cudaStream_t stream);

// Modelled time (microseconds) of the products kernel of this layer on `pairs`
// CTA pairs, and of its projection kernel on `ctas` SMs (both from B200
// measurements); lbp_backward_batch balances the two when it runs the
// projection of one layer beside the products kernel of another.
double fused_products_model_us(const lbp_layer& L, const BasisPlan& bp, int pairs);
// The plan of a call on `units` CTAs or CTA pairs; bp null: exact backpropagation.  `shape`
// receives what was planned.
const TilePlan& fused_tile_plan(const lbp_layer& L, const BasisPlan* bp, int n_extra, size_t planes_bytes, int units,
                                bool pair, PlanShape* shape);
double fused_projection_model_us(const lbp_layer& L, const BasisPlan& bp, int ctas);

// Whether the products kernel runs on CTA pairs (tcgen05 cta_group::2): Cin >= 128
// and an even SM count.
bool fused_pair_supported(const lbp_layer& L, int sms);

}  // namespace lbp
