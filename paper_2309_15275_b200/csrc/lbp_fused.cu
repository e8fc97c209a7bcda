// Persistent kernel for the two products of Algorithm 1 (bf16 data) with the
// expansion in its epilogue, run after the projection kernel; also both products of
// exact backpropagation (Eq. 2).
//
// A unit works through a static list of output tiles of the two products, fp32
// accumulators in TMEM, operands fed by TMA.  A unit is a pair of CTAs on
// neighbouring SMs sharing one tile through tcgen05.mma.cta_group::2 (each CTA
// loads its own 128 rows of A and half of B, the tensor cores of both SMs read the
// two halves from both shared memories: a third less operand traffic per SM, and
// operand delivery from L2 is what bounds these products), or, on narrow layers
// and odd SM counts, a single CTA.
//
//   GW tile (i, j):  g_W[rows i, BNw j ..] = g_y_hat^T x_hat          K = all low-rank rows
//   GX tile (m, n):  g_x_hat^T[channels n, rows m] = W^T g_y_hat^T    K = Cout
//
// Rows of A per CTA: 128 rows of g_W (GW) or 128 channels (GX).  GX is computed
// transposed, channels along the TMEM lanes, so that a thread of the epilogue holds
// every coefficient of a block for its channel: it applies the transposed bases
// (Eq. 7) in registers and g_x_hat never leaves the chip.  The low-rank rows lie
// along N: a tile takes as many whole blocks as fit its BNx columns, wherever they
// start, so the coefficient matrices are dense.  Tokens outside the grid (class
// tokens; all tokens in exact backpropagation) are further k-blocks of every GW
// tile and GX tiles of their own, read through tensor maps of their own where they
// lie.
//
// Warp roles: warp 0 TMA producer, warp 1 TMEM owner and tcgen05 issuer (the
// leader CTA's of a pair), warps 2 and 3 the TMA stores of the two epilogue groups,
// warps 4-19 epilogue in two groups of eight that take turns on the blocks (GX) or
// 32-column chunks (GW) of a tile, while the tensor core already works on the next
// tile (two accumulator slots in TMEM, used alternately).
// All roles walk the same tile list.  Barriers:
//   full[s]      leader's; its producer expects the bytes of both CTAs, and the
//                TMA loads of both CTAs complete on it (.cta_group::2 loads)
//   empty[s]     one per CTA; tcgen05.commit multicasts to both
//   acc_full[t]  one per CTA; commit multicasts to both
//   acc_empty[t] leader's; the epilogue warps of both CTAs arrive on it
//   fill_full / fill_empty: buffers between an epilogue group and its store warp
// No cluster-multicast load is used.  Every wait is bounded and an expired wait is
// reported through the status block.
#include <cuda_bf16.h>

#include <cstdio>
#include <cstdlib>

#include "lbp_fused.cuh"
#include "lbp_fused_epilogue.cuh"
#include "lbp_internal.h"
#include "ptx_sm100.cuh"
#include "wht_device.cuh"

namespace lbp {
namespace fused {

constexpr int BK = 64;
constexpr int kABytes = BM * BK * 2;             // 16 KB: this CTA's 128 rows of A
constexpr int kBBytes = 128 * BK * 2;            // 16 KB: this CTA's half of B (a pair's), or up to 128 columns
constexpr int kStageBytes = kABytes + kBBytes;   // 32 KB
constexpr int kChunkBytes = 64 * BK * 2;         // 8 KB: one 64-wide chunk of an MN-major tile
// warps 0-3: TMA producer, tensor-core issuer, a store warp per epilogue group; then those groups
constexpr int kThreads = (4 + 8 * kEGroups) * 32;
constexpr int kStages = 5;
constexpr int kOffBar = kStages * kStageBytes + kEGroups * kGroupBytes;   // ring, buffers, then the barriers
constexpr int kSmemBytes = kOffBar + 384 + 1024;
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget of one CTA exceeded");
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kSlotCols = 256;   // two accumulator slots; tile number t of a unit uses slot t & 1

// Tensor maps of the operands: g_y_hat as GX B (rows x 64 k) and as GW A, x_hat, W;
// g_y and x of the tokens outside the grid in the same roles.  Where a call has no
// grid, or no such tokens, the maps of that part are copies of the other's (unused).
struct OperandMaps {
  CUtensorMap gyhat_k, gyhat_mn, xhat, w;
  CUtensorMap gye_k, gye_mn, xe;
};

// ---- PTX of the CTA-pair forms ------------------------------------------------
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// shared::cluster address of `local_smem_addr` in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_rank(uint32_t local_smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_smem_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// TMA load whose completion is signalled on a barrier that may live in the peer CTA
// `policy`: L2 eviction hint (the operands are read by several units, from L2)
__device__ __forceinline__ void tma_load_2d_pair(void* smem_dst, const CUtensorMap* m,
                                                 uint32_t bar_cluster_addr, int32_t x, int32_t y,
                                                 uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(ptx::smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(bar_cluster_addr), "r"(x), "r"(y), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   ptx::smem_u32(smem_dst)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void mma_bf16_ss_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                                 uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrive on the barrier at the same shared-memory offset in both CTAs of the pair
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar) {
  const uint16_t mask = 3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 "
      "[%0], %1;" ::"r"(ptx::smem_u32(bar)),
      "h"(mask)
      : "memory");
}

// Role timeline (diagnostic builds only): slot 0 kernel start, 2 producer done,
// 3 MMA issuer done, 4 epilogue done, from 8 on eight slots per tile.
__device__ __forceinline__ void trace_mark(const FusedParams& p, int slot) {
#ifdef LBP_ROLE_TRACE
  if (p.trace != nullptr) {
    unsigned long long now;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now));
    atomicMax(p.trace + blockIdx.x * kTraceSlots + slot, now);
  }
#else
  (void)p, (void)slot;
#endif
}

// ------------------------------------------------------------------ kernel ----
template <int K, int CORE, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
    lbp_products_kernel(const __grid_constant__ OperandMaps tm, const __grid_constant__ StoreMaps sm,
                        const __grid_constant__ FusedParams p, const __grid_constant__ FusedBasis fb,
                        const __grid_constant__ FusedSchedule sc) {
  using X = Expand<K, CORE>;
  constexpr int kBufs = X::kBufs;
  static_assert((2 * kStages + 4 + 2 * kEGroups * kBufs) * 8 + 8 <= 384, "barriers");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + kOffBar);
  uint64_t* empty_bar = full_bar + kStages;
  uint64_t* acc_full = empty_bar + kStages;                   // [2]
  uint64_t* acc_empty = acc_full + 2;                         // [2], the leader's are used
  uint64_t* fill_full = acc_empty + 2;                        // [kEGroups][kBufs]
  uint64_t* fill_empty = fill_full + kEGroups * kBufs;    // [kEGroups][kBufs]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fill_empty + kEGroups * kBufs);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  constexpr int kCtas = PAIR ? 2 : 1;   // CTAs of a unit
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = PAIR ? static_cast<int>(cluster_ctarank()) : 0;
  const int unit = blockIdx.x / kCtas, units = gridDim.x / kCtas;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(&full_bar[s], 1);
      ptx::mbar_init(&empty_bar[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      ptx::mbar_init(&acc_full[s], 1);
      ptx::mbar_init(&acc_empty[s], kCtas * 8 * kEGroups);   // epilogue warps of all CTAs of the unit
    }
    for (int s = 0; s < kEGroups * kBufs; ++s) {
      ptx::mbar_init(&fill_full[s], 8);    // the warps of the group
      ptx::mbar_init(&fill_empty[s], 1);   // its store warp
    }
    ptx::mbar_fence_init();
    *abort_flag = 0;
    ptx::prefetch_tensormap(&tm.gyhat_k);
    ptx::prefetch_tensormap(&tm.gyhat_mn);
    ptx::prefetch_tensormap(&tm.xhat);
    ptx::prefetch_tensormap(&tm.w);
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      tmem_alloc_pair(tmem_slot, kTmemCols);
      tmem_relinquish_pair();
    } else {
      ptx::tmem_alloc(tmem_slot, kTmemCols);
      ptx::tmem_relinquish();
    }
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();   // the peer's barriers exist before anything is signalled on them
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  const int my_tiles = unit_tile_count(p, sc, unit, units);
  if (threadIdx.x == 0) trace_mark(p, 0);

  if (warp == 0) {
    // =========================== TMA producer ===========================
    if (ptx::elect_one()) {
      // launched with programmatic stream serialization: x_hat / g_y_hat of the
      // projection kernel may only be read after this wait
      asm volatile("griddepcontrol.wait;" ::: "memory");
      // The next kernel on the stream may be scheduled as SMs free up.  A projection that
      // defers its own wait (buffers disjoint from this kernel's) then reads x and g_y at
      // once, so this may be said only after whatever lies ahead has completed.
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
      const uint64_t keep = ptx::l2_policy_evict_last();
      uint32_t it = 0;
      bool ok = true;
      for (int ti = 0; ti < my_tiles && ok && !p.test_stall; ++ti) {
        const WorkTile tl = unit_tile(p, sc, unit, units, ti);
        const int part = (tl.is_gw ? p.BNw : p.BNx) / kCtas;   // this CTA's share of B's columns
        const uint32_t tx = static_cast<uint32_t>(kCtas * (kABytes + part * BK * 2));
        for (int kb = tl.kb0; kb < tl.kb0 + tl.n_kb; ++kb) {
          const int s = static_cast<int>(it % kStages);
          if (!ptx::mbar_wait(&empty_bar[s], ((it / kStages) + 1) & 1u, p.status, (5u << 16) | 1u)) {
            ok = false;
            break;
          }
          uint8_t* sa = smem + s * kStageBytes;
          uint8_t* sb = sa + kABytes;
          if (rank == 0) ptx::mbar_expect_tx(&full_bar[s], tx);
          uint32_t bar = 0;
          if constexpr (PAIR) bar = map_to_rank(ptx::smem_u32(&full_bar[s]), 0);
          auto load = [&](void* dst, const CUtensorMap& m, int x, int y) {
            if constexpr (PAIR)
              tma_load_2d_pair(dst, &m, bar, x, y, keep);
            else
              ptx::tma_load_2d_hint(dst, &m, &full_bar[s], x, y, keep);
          };
          if (tl.is_gw) {
            // A = g_y_hat^T: stored (rows, Cout), MN-major; past the low-rank rows
            // come those of the tokens outside the grid
            const bool ext = kb >= p.kb_lr;
            const CUtensorMap& ma = ext ? tm.gye_mn : tm.gyhat_mn;
            const CUtensorMap& mb = ext ? tm.xe : tm.xhat;
            const int y = (ext ? kb - p.kb_lr : kb) * BK;
            const int m0 = (tl.a * kCtas + rank) * BM;
            load(sa, ma, m0, y);
            load(sa + kChunkBytes, ma, m0 + 64, y);
            const int n0 = tl.b * p.BNw + rank * part;
            for (int c = 0; c < part / 64; ++c) load(sb + c * kChunkBytes, mb, n0 + c * 64, y);
          } else {
            // A = W^T: stored (Cout, Cin), MN-major; B = g_y_hat rows, K-major
            const int m0 = (tl.b * kCtas + rank) * BM;
            load(sa, tm.w, m0, kb * BK);
            load(sa + kChunkBytes, tm.w, m0 + 64, kb * BK);
            const bool ext = tl.a >= p.n_rt;
            const int n0 = ext ? (tl.a - p.n_rt) * p.BNx : tl.a * p.bpt * p.r;
            load(sb, ext ? tm.gye_k : tm.gyhat_k, kb * BK, n0 + rank * part);
          }
          ++it;
        }
      }
      if (!ok) *abort_flag = 1;
      trace_mark(p, 2);
    }
  } else if (warp == 1) {
    // =========================== tcgen05 issuer (leader only) ===========================
    if (rank == 0 && ptx::elect_one()) {
      uint32_t it = 0;
      bool ok = true;
      const uint32_t idesc_w = ptx::idesc_bf16(kCtas * BM, p.BNw, true, true);
      const uint32_t idesc_x = ptx::idesc_bf16(kCtas * BM, p.BNx, true, false);
      auto commit = [](uint64_t* bar) {
        if constexpr (PAIR)
          mma_commit_pair(bar);
        else
          ptx::mma_commit(bar);
      };
      for (int ti = 0; ti < my_tiles && ok; ++ti) {
        const WorkTile tl = unit_tile(p, sc, unit, units, ti);
        const int slot = ti & 1;
        const uint32_t d_tmem = tmem_base + slot * kSlotCols;
        const uint32_t idesc = tl.is_gw ? idesc_w : idesc_x;
        const uint32_t uses = static_cast<uint32_t>(ti >> 1);   // earlier uses of this slot
        // the accumulator slot must have been drained by the epilogue
        if (!ptx::mbar_wait(&acc_empty[slot], (uses + 1) & 1u, p.status, (5u << 16) | 4u)) {
          ok = false;
          break;
        }
        for (int kb = 0; kb < tl.n_kb; ++kb) {
          const int s = static_cast<int>(it % kStages);
          if (!ptx::mbar_wait(&full_bar[s], (it / kStages) & 1u, p.status, (5u << 16) | 3u)) {
            ok = false;
            break;
          }
          if (kb == 0 && ti < 15) trace_mark(p, 8 + 8 * ti);
          ptx::tc_fence_after_sync();
          const uint32_t sa = ptx::smem_u32(smem + s * kStageBytes);
          const uint32_t sb = sa + kABytes;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            // A MN-major (16 k = 16 rows of 128 bytes further per step); B MN-major
            // (GW) or K-major (GX: 16 k = 32 bytes further)
            const uint64_t da = ptx::smem_desc_sw128(sa + kk * 2048, kChunkBytes, 1024);
            const uint64_t db = tl.is_gw ? ptx::smem_desc_sw128(sb + kk * 2048, kChunkBytes, 1024)
                                         : ptx::smem_desc_sw128(sb + kk * 32, 16, 1024);
            const uint32_t add = (kb == 0 && kk == 0) ? 0u : 1u;
            if constexpr (PAIR)
              mma_bf16_ss_pair(d_tmem, da, db, idesc, add);
            else
              ptx::mma_bf16_ss(d_tmem, da, db, idesc, add);
          }
          commit(&empty_bar[s]);
          ++it;
        }
        if (!ok) break;
        commit(&acc_full[slot]);
        if (ti < 15) trace_mark(p, 8 + 8 * ti + 1);
      }
      if (!ok) *abort_flag = 1;
      trace_mark(p, 3);
    }
  } else {
    // ============ epilogue (each CTA its own 128 lanes): two groups of eight warps (from
    // warp 4 on), each with a store warp (warps 2 and 3) ============
    const bool stores = warp < 4;
    const int eg = stores ? warp - 2 : (warp - 4) >> 3;
    const int sub = (warp >> 2) & 1 ? 0 : 1;             // half of the group (warps 4-7 and 12-15: 0)
    const int quarter = warp & 3;                        // TMEM lane quarter this warp may read
    const bool first = sub == 0 && quarter == 0 && lane == 0;   // one thread of the group
    const int bar_id = 1 + eg;                           // the group; its halves: 3 + 2 eg + sub
    Fills<X> fills{smem + kStages * kStageBytes + eg * kGroupBytes, fill_full + eg * kBufs,
                       fill_empty + eg * kBufs, p.status, 0u, 0u};
    bool alive = true;
    for (int ti = 0; ti < my_tiles && alive; ++ti) {
      const WorkTile tl = unit_tile(p, sc, unit, units, ti);
      const int slot = ti & 1;
      DrainTile dt;
      dt.row_base = ((tl.is_gw ? tl.a : tl.b) * kCtas + rank) * BM;
      dt.row_tile = tl.a;
      dt.col_base = tl.b * p.BNw;
      dt.slice = tl.slice;
      dt.tmem_acc = tmem_base + slot * kSlotCols;
      if (stores) {
        if (!tl.is_gw) alive = store_gx<K, CORE>(p, sm, dt, fills, eg, lane);
        // before a GW tile, which uses the buffers its own way: everything has been read
        if (alive && !tl.is_gw && ti + 1 < my_tiles && unit_tile(p, sc, unit, units, ti + 1).is_gw)
          fills.flush(lane);
        continue;
      }
      bool ok = ptx::mbar_wait(&acc_full[slot], static_cast<uint32_t>(ti >> 1) & 1u, p.status, (5u << 16) | 5u);
      // a GW tile stages its chunks in the buffers: the stores of every fill have been read
      if (tl.is_gw)
        for (int b = 0; b < kBufs && ok; ++b) ok = fills.wait_empty(fills.count + b);
      // One answer for the whole group: a thread that saw its own wait expire, or
      // the flag another role raised, takes the other 255 threads with it (read
      // one by one after the barrier, the flag could split the group, and the
      // threads left inside the tile would wait on a barrier that never fills).
      if (named_bar_or(bar_id, 256, !ok || *abort_flag != 0)) {
        if (first) *abort_flag = 1;
        break;
      }
      ptx::tc_fence_after_sync();
      if (first && ti < 15) trace_mark(p, 8 + 8 * ti + 2 + 2 * eg);
      uint64_t* const mine = &acc_empty[slot];
      auto release = [mine]() {
        if constexpr (PAIR)
          mbar_arrive_cluster(map_to_rank(ptx::smem_u32(mine), 0));
        else
          ptx::mbar_arrive(mine);
      };
      bool drained = true;
      if (tl.is_gw)
        drain_gw(p, dt, reinterpret_cast<float*>(fills.buf + sub * kGwStageBytes), 3 + 2 * eg + sub,
                 2 * eg + sub, quarter, lane, release);
      else if (tl.a >= p.n_rt)
        drained = drain_gx_extra(p, dt, fills, eg, sub, quarter, lane, release);
      else
        drained = drain_gx<K, CORE>(p, fb, dt, fills, eg, sub, quarter, lane, release);
      if (!drained) *abort_flag = 1;   // the group leaves together at the next tile
      if (first && ti < 15) {
        trace_mark(p, 8 + 8 * ti + 3 + 2 * eg);
#ifdef LBP_ROLE_TRACE
        if (eg == 0 && p.trace != nullptr)
          p.trace[blockIdx.x * kTraceSlots + 8 + 8 * ti + 6] =
              (static_cast<unsigned long long>(tl.is_gw) << 32) | static_cast<unsigned>(tl.n_kb);
#endif
      }
    }
    if (stores) {
      if (!alive) *abort_flag = 1;
      bulk_wait_all();   // this warp's stores are complete before the CTA leaves
    }
    if (first && !stores) trace_mark(p, 4);   // latest of the groups
  }

  ptx::tc_fence_before_sync();
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();   // neither CTA leaves while the other may still touch its memory
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    if constexpr (PAIR)
      tmem_dealloc_pair(tmem_base, kTmemCols);
    else
      ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
}

}  // namespace fused

// --------------------------------------------------------------- launcher ----
static thread_local const FusedOverlap* g_overlap = nullptr;
void set_fused_overlap(const FusedOverlap* ov) { g_overlap = ov; }
const FusedOverlap* fused_overlap() { return g_overlap; }

static thread_local bool g_test_stall = false;
void set_test_stall(bool on) { g_test_stall = on; }
bool test_stall() { return g_test_stall; }
static thread_local bool g_test_stall_projection = false;
void set_test_stall_projection(bool on) { g_test_stall_projection = on; }
bool test_stall_projection() { return g_test_stall_projection; }

static long long grid_blocks(const lbp_layer& L) {
  return static_cast<long long>(L.B) * blocks_along(L.H, L.k) * blocks_along(L.W, L.k);
}

bool fused_supported(const lbp_layer& L, const BasisPlan& bp) {
  return L.dtype == LBP_BF16 && grid_blocks(L) * bp.r < (1ll << 31) - 256 &&
         (L.k == 4 || L.k == 8 || L.k == 16) && bp.r <= fused_max_rank(L.k) && bp.LB <= 8 && bp.LB <= L.k;
}

bool fused_pair_supported(const lbp_layer& L, int sms) {
  if (!tune_options().pair) return false;
  return L.Cin >= 128 && sms >= 2 && (sms % 2) == 0;
}

size_t fused_scratch_bytes(const lbp_layer& L, int r, FusedLayout* lay) {
  const long long rows = grid_blocks(L) * r;
  FusedLayout l;
  size_t off = 0;
  l.x_hat = off;
  off += static_cast<size_t>(rows) * L.Cin * 2;
  off = (off + 1023) / 1024 * 1024;
  l.gy_hat = off;
  off += static_cast<size_t>(rows) * L.Cout * 2;
  off = (off + 1023) / 1024 * 1024;
  // fp32 planes for K slices of g_W: only layers with few GW tiles slice, and
  // slices * tiles stays below the SM count (bounded here for up to 256 SMs)
  l.planes = off;
  {
    const long long tiles_min = ((L.Cout + 127) / 128) * ((L.Cin + 255) / 256);
    long long s_cap = tiles_min >= 96 ? 1 : 192 / tiles_min;
    const long long kbs = (rows + fused::BK - 1) / fused::BK;
    if (s_cap > kbs) s_cap = kbs;
    l.planes_bytes = s_cap > 1 ? static_cast<size_t>(s_cap) * L.Cout * L.Cin * 4 : 0;
    const size_t cap = 48u << 20;
    if (l.planes_bytes > cap) l.planes_bytes = cap;
  }
  off += l.planes_bytes;
  off = (off + 1023) / 1024 * 1024;
  l.trace = off;
  off += kFusedTraceBytes;
  l.total = (off + 1023) / 1024 * 1024;
  if (lay) *lay = l;
  return l.total;
}

// The form of the expansion a basis plan takes (see Expand): rank 1 is a 2 x 2 array
// with three empty places.
static int expand_core(const BasisPlan& bp) {
  if (bp.LB < 8) return bp.LB < 2 ? 2 : bp.LB;
  int hl = 0, lh = 0, hh = 0;
  for (int q = 0; q < bp.r; ++q) {
    const bool hi = bp.seq_i[q] >= 4, hj = bp.seq_j[q] >= 4;
    hl += hi && !hj;
    lh += hj && !hi;
    hh += hi && hj;
  }
  if (hh > 0) return 8;
  return hl <= 1 && lh <= 1 ? fused::kCoreSparse : fused::kCoreNoHH;
}

// The same bases with their slots ordered by rows (i, then j).  Only where every row
// holds j = 0 .. n_i - 1 (true of every set that contains, with a basis, all those of
// lower frequency along W: the LP_L1, LP_Linf and PREFIX sets): the expansion then
// reads a row with one load.  False: bp is not changed.
static bool order_by_rows(BasisPlan* bp) {
  int slot_of[8][8], n[8] = {};
  for (auto& row : slot_of)
    for (int& q : row) q = -1;
  for (int q = 0; q < bp->r; ++q) {
    if (bp->seq_i[q] >= 8 || bp->seq_j[q] >= 8) return false;
    slot_of[bp->seq_i[q]][bp->seq_j[q]] = q;
    ++n[bp->seq_i[q]];
  }
  for (int i = 0; i < 8; ++i)
    for (int j = 0; j < n[i]; ++j)
      if (slot_of[i][j] < 0) return false;
  const BasisPlan old = *bp;
  int16_t new_slot[kMaxRank];
  int q = 0;
  for (int i = 0; i < 8; ++i)
    for (int j = 0; j < n[i]; ++j, ++q) {
      const int from = slot_of[i][j];
      new_slot[from] = static_cast<int16_t>(q);
      bp->nat_i[q] = old.nat_i[from];
      bp->nat_j[q] = old.nat_j[from];
      bp->seq_i[q] = old.seq_i[from];
      bp->seq_j[q] = old.seq_j[from];
    }
  for (int p = 0; p < bp->LB * bp->LB; ++p)
    if (old.qmap[p] >= 0) bp->qmap[p] = new_slot[old.qmap[p]];
  return true;
}

static FusedBasis make_fused_basis(const BasisPlan& bp, int core, bool by_rows) {
  FusedBasis fb{};
  fb.by_rows = by_rows ? 1 : 0;
  if (by_rows)
    for (int q = bp.r - 1; q >= 0; --q) fb.row[bp.seq_i[q]] = q;
  if (core <= 4) {
    for (int a = 0; a < bp.LB; ++a)
      for (int b = 0; b < bp.LB; ++b) {
        const int q = bp.qmap[a * bp.LB + b];
        fb.col[a * core + b] = q >= 0 ? q : 0;
        fb.keep[a * core + b] = q >= 0 ? 0xffffffffu : 0u;
      }
    return fb;
  }
  for (int a = 0; a < 8; ++a)
    for (int b = 0; b < 8; ++b) {
      const int q = bp.qmap[a * 8 + b];
      if (q < 0) continue;
      // bit 0 of a natural index is set exactly where the sequency is 4 or more
      const int quad = 2 * (b & 1) + (a & 1), pos = (a >> 1) * 4 + (b >> 1);
      if (core == fused::kCoreSparse && quad != 0) {
        const int side = quad - 1;
        fb.ex_col[side] = q;
        fb.ex_keep[side] = 0xffffffffu;
        for (int i = 0; i < 16; ++i) {
          const int par = __builtin_popcount((a >> 1) & (i >> 2)) + __builtin_popcount((b >> 1) & (i & 3));
          fb.ex_sign[side][i] = (par & 1) != 0 ? -1.f : 1.f;
        }
      } else {
        fb.col[quad * 16 + pos] = q;
        fb.keep[quad * 16 + pos] = 0xffffffffu;
      }
    }
  return fb;
}

// blocks * piece low-rank rows; blocks = 0: exact backpropagation on n_extra tokens
static PlanShape plan_shape(const lbp_layer& L, long long blocks, int piece, int core, int n_extra,
                            size_t planes_bytes, int units, bool pair) {
  PlanShape s{};
  s.gw_rows = L.Cout;
  s.gw_cols = L.Cin;
  s.gx_side = L.Cin;
  s.blocks = static_cast<int>(blocks);
  s.piece = piece;
  s.n_extra = n_extra;
  s.units = units;
  s.pair = pair ? 1 : 0;
  s.bnw_step = pair ? 128 : 64;
  s.bnx_step = 32;
  s.bn_max = pair ? 256 : 128;
  s.max_splits = static_cast<int>(planes_bytes / (static_cast<size_t>(L.Cout) * L.Cin * 4));
  s.expand_bytes = blocks > 0 ? L.k * L.k * 2 : 2;
  s.epi_kind = blocks == 0 ? -1 : core <= 4 ? 0 : core == fused::kCoreSparse ? 1 : 2;
  s.num_kb_w = static_cast<int>((blocks * piece + fused::BK - 1) / fused::BK) +
               (n_extra + fused::BK - 1) / fused::BK;
  s.num_kb_x = (L.Cout + fused::BK - 1) / fused::BK;
  return s;
}

const TilePlan& fused_tile_plan(const lbp_layer& L, const BasisPlan* bp, int n_extra, size_t planes_bytes, int units,
                                bool pair, PlanShape* shape) {
  *shape = bp != nullptr ? plan_shape(L, grid_blocks(L), bp->r, expand_core(*bp), n_extra, planes_bytes, units, pair)
                         : plan_shape(L, 0, 1, 4, n_extra, planes_bytes, units, pair);
  return plan_products(*shape);
}

double fused_products_model_us(const lbp_layer& L, const BasisPlan& bp, int pairs) {
  FusedLayout lay;
  fused_scratch_bytes(L, bp.r, &lay);
  // measured times sit a little above the model, plus the launch and the first
  // operand tiles
  return 1.1 * plan_products(plan_shape(L, grid_blocks(L), bp.r, expand_core(bp), 0, lay.planes_bytes,
                                         pairs, true))
                    .model_us +
         4.0;
}

double fused_projection_model_us(const lbp_layer& L, const BasisPlan& bp, int ctas) {
  const double T = static_cast<double>(L.B) * L.H * L.W;
  const double nb = static_cast<double>(grid_blocks(L));
  const double bytes = 2.0 * (T + nb * bp.r) * (L.Cin + L.Cout);
  // one SM moves about 80 GB/s in and out, the chip about 5.3 TB/s
  const double rate = ctas * 80e3 < 5.3e6 ? ctas * 80e3 : 5.3e6;   // bytes per microsecond
  return bytes / rate + 5.0;
}

// Algorithm 1, steps 1-2: x_hat and g_y_hat (g_y_hat alone when x_hat is given).
static int fused_project(const void* x, void* x_hat, const void* g_y, void* gy_hat, const lbp_layer& L,
                         const BasisPlan& bp, const CallViews* views, uint32_t* status,
                         cudaStream_t stream) {
  const FusedOverlap* ov = fused_overlap();
  cudaStream_t ps = ov != nullptr ? ov->proj_stream : stream;
  if (ov != nullptr) set_projection_launch(ProjLaunch{ov->proj_ctas, ov->proj_ctas > 0, false});
  const float sgy = fused_scale_gy(L.k, x == nullptr);
  int e = LBP_OK;
  if (x != nullptr)
    e = launch_project2(g_y, gy_hat, L.Cout, x, x_hat, L.Cin, LBP_BF16, L.B, L.H, L.W, bp, status,
                        ps, sgy, fused_scale_x(L.k), views ? &views->gy : nullptr,
                        views ? &views->x : nullptr);
  else
    e = launch_project(g_y, gy_hat, LBP_BF16, L.B, L.H, L.W, L.Cout, bp, status, ps, sgy,
                       views ? &views->gy : nullptr);
  if (ov != nullptr) {
    set_projection_launch(ProjLaunch{0, false, true});
    if (e != LBP_OK) return e;
    LBP_CUDA_TRY(cudaEventRecord(ov->proj_done, ps));
    LBP_CUDA_TRY(cudaStreamWaitEvent(stream, ov->proj_done, 0));
  }
  return e;
}

// Maps of the expansion's stores: map du * S + dv addresses the tokens (S u + du,
// S v + dv) of every image, so that its extents clip exactly at the grid's edge.
// Maps of offsets a small grid does not have are never used (copies of the first).
static int encode_store_maps(fused::StoreMaps* sm, void* g_x, const lbp_layer& L, int S, int T, int box_rows,
                             const lbp_view& v) {
  for (int du = 0; du < S; ++du)
    for (int dv = 0; dv < S; ++dv) {
      if (du >= L.H || dv >= L.W) {
        sm->m[du * S + dv] = sm->m[0];
        continue;
      }
      const lbp_view s{v.image, v.row * S, v.token * S};
      __nv_bfloat16* base = static_cast<__nv_bfloat16*>(g_x) + du * v.row + dv * v.token;
      if (int e = encode_box_tensor_map(&sm->m[du * S + dv], base, LBP_BF16, L.B, (L.H - du + S - 1) / S,
                                        (L.W - dv + S - 1) / S, L.Cin, 128, T, box_rows, false, &s))
        return e;
    }
  return LBP_OK;
}

// One launch of the products kernel.
struct ProductsCall {
  const lbp_layer* L;
  // the grid's part; blocks = 0: none
  long long blocks;
  int r, core;
  const void *gy_hat, *x_hat;
  void* g_x;
  lbp_view gx_view;
  float gx_scale;
  FusedBasis fb;
  // the tokens outside the grid; ex.n_extra = 0: none
  FusedExtras ex;
  const void* W;
  void* g_W;
  float* planes;
  size_t planes_bytes;
  uint32_t* status;
#ifdef LBP_ROLE_TRACE
  unsigned long long* trace;
#endif
};

template <int K, int CORE, bool PAIR>
static int launch_kernel(const cudaLaunchConfig_t& cfg, const fused::OperandMaps& tm, const fused::StoreMaps& sm,
                         const FusedParams& p, const FusedBasis& fb, const FusedSchedule& sc) {
  auto kern = fused::lbp_products_kernel<K, CORE, PAIR>;
  static PerDevice configured;
  if (int e = allow_dynamic_smem(configured, reinterpret_cast<const void*>(kern), fused::kSmemBytes)) return e;
  LBP_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, tm, sm, p, fb, sc));
  count_launch();
  return LBP_OK;
}

static int launch_products(const ProductsCall& c, cudaStream_t stream) {
  using namespace fused;
  const lbp_layer& L = *c.L;
  const int K = L.k, n_extra = c.ex.n_extra;
  int dev = 0, sms = 0;
  LBP_CUDA_TRY(cudaGetDevice(&dev));
  LBP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const bool pair = fused_pair_supported(L, sms);
  const FusedOverlap* ov = fused_overlap();
  int units = pair ? sms / 2 : sms;
  if (pair && ov != nullptr && ov->prod_units > 0 && ov->prod_units < units) units = ov->prod_units;

  const TilePlan& plan =
      plan_products(plan_shape(L, c.blocks, c.r, c.core, n_extra, c.planes_bytes, units, pair));
  const int ctas = pair ? 2 : 1;
  FusedParams p{};
  p.nb = static_cast<int32_t>(c.blocks);
  p.Hb = blocks_along(L.H, K);
  p.Wb = blocks_along(L.W, K);
  p.H = L.H;
  p.W = L.W;
  p.r = c.r;
  p.Cin = L.Cin;
  p.Cout = L.Cout;
  p.BNx = plan.BNx;
  p.bpt = plan.bpt;
  p.n_ct = (L.Cin + ctas * BM - 1) / (ctas * BM);
  p.n_rt = (p.nb + p.bpt - 1) / p.bpt;
  p.num_kb_x = (L.Cout + BK - 1) / BK;
  p.n_gx_tiles = p.n_ct * (p.n_rt + (n_extra + p.BNx - 1) / p.BNx);
  const long long rows = c.blocks * c.r;
  p.BNw = plan.BNw;
  p.mt_w = (L.Cout + ctas * BM - 1) / (ctas * BM);
  p.nt_w = (L.Cin + p.BNw - 1) / p.BNw;
  p.kb_lr = static_cast<int>((rows + BK - 1) / BK);
  p.num_kb_w = p.kb_lr + (n_extra + BK - 1) / BK;
  p.gw_splits = plan.splits;
  p.kb_per_split_w = plan.kbps;
  p.n_gw_tiles = p.mt_w * p.nt_w * p.gw_splits;
  p.gw_planes = c.planes;
  p.gw_bf16 = L.gw_dtype == LBP_BF16 ? 1 : 0;
  p.beta = c.ex.beta;
  p.gx_scale = c.gx_scale;
  p.n_extra = n_extra;
  p.g_W = c.g_W;
  p.status = c.status;
  p.test_stall = test_stall() ? 1 : 0;
#ifdef LBP_ROLE_TRACE
  p.trace = c.trace;
  if (p.trace != nullptr) LBP_CUDA_TRY(cudaMemsetAsync(p.trace, 0, kFusedTraceBytes, stream));
#endif

  OperandMaps tm;
  StoreMaps sm;
  const int T = c.core <= 4 ? 4 : 8;
  if (int e = encode_matrix_tensor_map(&tm.w, c.W, L.Cout, L.Cin, BK)) return e;
  if (rows > 0) {
    if (int e = encode_matrix_tensor_map(&tm.gyhat_k, c.gy_hat, rows, L.Cout, p.BNx / ctas)) return e;
    if (int e = encode_matrix_tensor_map(&tm.gyhat_mn, c.gy_hat, rows, L.Cout, BK)) return e;
    if (int e = encode_matrix_tensor_map(&tm.xhat, c.x_hat, rows, L.Cin, BK)) return e;
    if (int e = encode_store_maps(&sm, c.g_x, L, K / T, T, 4, c.gx_view)) return e;
  }
  if (n_extra > 0) {
    if (int e = encode_matrix_tensor_map(&tm.gye_k, c.ex.gy, n_extra, L.Cout, p.BNx / ctas, c.ex.gy_pitch)) return e;
    if (int e = encode_matrix_tensor_map(&tm.gye_mn, c.ex.gy, n_extra, L.Cout, BK, c.ex.gy_pitch)) return e;
    if (int e = encode_matrix_tensor_map(&tm.xe, c.ex.x, n_extra, L.Cin, BK, c.ex.x_pitch)) return e;
    const int64_t pitch = c.ex.gx_pitch > 0 ? c.ex.gx_pitch : L.Cin;
    const lbp_view rows_view{pitch * n_extra, pitch * n_extra, pitch};
    if (int e = encode_box_tensor_map(&sm.extra, c.ex.gx, LBP_BF16, 1, 1, n_extra, L.Cin, 128, 32, 1, false,
                                      &rows_view))
      return e;
  } else {
    tm.gye_k = tm.gyhat_k;
    tm.gye_mn = tm.gyhat_mn;
    tm.xe = tm.xhat;
    sm.extra = sm.m[0];
  }
  if (rows == 0) {
    tm.gyhat_k = tm.gye_k;
    tm.gyhat_mn = tm.gye_mn;
    tm.xhat = tm.xe;
    for (CUtensorMap& m : sm.m) m = sm.extra;
  }

  const int total_tiles = p.n_gw_tiles + p.n_gx_tiles;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas * (total_tiles < units ? total_tiles : units));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  unsigned n_attr = 0;
  if (pair) {
    attr[n_attr].id = cudaLaunchAttributeClusterDimension;
    attr[n_attr].val.clusterDim.x = 2;
    attr[n_attr].val.clusterDim.y = 1;
    attr[n_attr++].val.clusterDim.z = 1;
  }
  // Beside a projection on another stream the kernel is launched in plain stream
  // order: launched early, its CTAs would sit on the SMs that projection is
  // meant to get while they wait for the kernel ahead.
  if (ov == nullptr) {
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr++].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n_attr;
  int e = LBP_ERR_BASIS;
#define LBP_CASE(KK, CC)                                                                          \
  case KK * 100 + CC:                                                                             \
    e = pair ? launch_kernel<KK, CC, true>(cfg, tm, sm, p, c.fb, plan.sched)                      \
             : launch_kernel<KK, CC, false>(cfg, tm, sm, p, c.fb, plan.sched);                    \
    break
  switch (K * 100 + c.core) {
    LBP_CASE(4, 2);
    LBP_CASE(4, 4);
    LBP_CASE(8, 2);
    LBP_CASE(8, 4);
    LBP_CASE(8, 6);
    LBP_CASE(8, 7);
    LBP_CASE(8, 8);
    LBP_CASE(16, 2);
    LBP_CASE(16, 4);
    LBP_CASE(16, 6);
    LBP_CASE(16, 7);
    LBP_CASE(16, 8);
  }
#undef LBP_CASE
  if (e != LBP_OK) return e;
  if (p.gw_splits > 1)
    return launch_splitk_reduce(p.gw_planes, c.g_W, static_cast<long long>(L.Cout) * L.Cin, p.gw_splits,
                                p.gw_bf16 != 0, p.beta, false, stream);
  return LBP_OK;
}

int launch_fused(const void* x, const void* x_hat_dense, const void* g_y, const void* W, void* g_x,
                 void* g_W, const lbp_layer& L, const BasisPlan& list, uint8_t* scratch,
                 uint32_t* status, cudaStream_t stream, FusedPhaseHook hook, void* hook_arg,
                 const CallViews* views, const FusedExtras* extras, int* dc_slot) {
  FusedLayout lay;
  fused_scratch_bytes(L, list.r, &lay);
  void* x_hat = scratch + lay.x_hat;
  void* gy_hat = scratch + lay.gy_hat;
  // the slots of a block may lie in any order as long as x_hat and g_y_hat agree;
  // coefficients handed in keep the caller's
  BasisPlan bp = list;
  const bool by_rows = x_hat_dense == nullptr && order_by_rows(&bp);
  if (int e = fused_project(x, x_hat, g_y, gy_hat, L, bp, views, status, stream)) return e;
  if (hook != nullptr)
    if (int e = hook(hook_arg, stream)) return e;
  ProductsCall c{};
  c.L = &L;
  c.blocks = grid_blocks(L);
  c.r = bp.r;
  c.core = expand_core(bp);
  c.gy_hat = gy_hat;
  c.x_hat = x_hat_dense != nullptr ? x_hat_dense : x_hat;
  c.g_x = g_x;
  c.gx_view = resolve_view(views ? &views->gx : nullptr, L.H, L.W, L.Cin);
  c.gx_scale = x_hat_dense != nullptr ? 1.0f / static_cast<float>(L.k) : 1.0f;
  c.fb = make_fused_basis(bp, c.core, by_rows);
  if (dc_slot != nullptr) {
    *dc_slot = -1;
    for (int q = 0; q < bp.r; ++q)
      if (bp.seq_i[q] == 0 && bp.seq_j[q] == 0) *dc_slot = q;
  }
  if (extras != nullptr) c.ex = *extras;
  c.W = W;
  c.g_W = g_W;
  c.planes = reinterpret_cast<float*>(scratch + lay.planes);
  c.planes_bytes = lay.planes_bytes;
  c.status = status;
#ifdef LBP_ROLE_TRACE
  c.trace = reinterpret_cast<unsigned long long*>(scratch + lay.trace);
#endif
  return launch_products(c, stream);
}

int launch_exact(const void* x, const void* g_y, const void* W, void* g_x, void* g_W, const lbp_layer& L,
                 long long tokens, float* planes, size_t planes_bytes, uint32_t* status,
                 cudaStream_t stream) {
  if (tokens >= (1ll << 31) - 256) return LBP_ERR_SHAPE;
  ProductsCall c{};
  lbp_layer Le = L;
  Le.k = 8;   // no grid: any instance of the kernel serves
  c.L = &Le;
  c.r = 1;
  c.core = 4;
  c.gx_scale = 1.f;
  c.ex.n_extra = static_cast<int>(tokens);
  c.ex.x = x;
  c.ex.gy = g_y;
  c.ex.gx = g_x;
  c.W = W;
  c.g_W = g_W;
  c.planes = planes;
  c.planes_bytes = planes_bytes;
  c.status = status;
  return launch_products(c, stream);
}

}  // namespace lbp
