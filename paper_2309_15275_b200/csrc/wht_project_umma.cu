// Projection of Eq. 6 on the tcgen05 tensor cores (bf16; orders 8 and 16 up to rank 48,
// order 4 at every rank).
//
//   t_hat[blk, q, c] = scale * sum_tok B_q[tok] * t[blk, tok, c]
//
// is a product of a block's tokens x channels with the +-1 basis matrix.  No warp
// touches the tile: a TMA box of 64 tokens x 64 channels lands in shared memory in the
// 128-byte-swizzled layout that is, as it lies, an MN-major A operand (m = channel,
// k = token); two boxes side by side make M = 128 channels.  B is the basis matrix,
// built once per CTA in shared memory (K-major, 16 to 64 rows: the r bases, the rest
// zero), so N follows the rank and four MMAs (128 x N x 16) take 16 KB of input.  With
// the data as B and the basis padded to M = 128, as this kernel had it before, the
// same input took 8 times the tensor-core work at r <= 16, about as much as the
// products of the layer themselves (and power is what bounds long runs).
//
// The chunks (a block x 64 channels) of both tensors are numbered through; an item is
// four consecutive ones, whatever block or tensor they belong to, so that narrow layers
// (48 channels: one chunk per block) fill the ring like wide ones.
//   order 8   a block is one box (8 x 8 tokens);
//   order 16  four parts of 64 tokens (four token rows each), every part a stage of its
//             own against its own 64 columns of the basis matrix, accumulating;
//   order 4   a "block" here is a strip of four along W, fetched as four boxes of 4 x 4
//             tokens: every MMA then contracts the 16 tokens of one block, into 16 columns
//             of its own.  (One 4 x 16 box has the four blocks' tokens in every MMA, zeros in
//             the basis matrix keeping them apart, and zero times the infinity of a block is
//             NaN in its neighbours; it took as long: 128 x 16 x 16 tokens of 3072 channels 48
//             us at rank 3, 57 at rank 8, 75 at rank 15.)
// The accumulator holds one channel per TMEM lane and one coefficient per column: a
// thread reads its r columns, rounds them and stores them to r rows of 64 channels in
// shared memory, from where one TMA store per chunk writes them.
//
// Roles: warps 0-3 TMA producers (one 64-channel chunk of an item each), warp 4 MMA
// issuer, warps 8-23 four epilogue warpgroups that take turns on the items (an item's
// epilogue is a chain of about a microsecond: two groups held an SM to 62 GB/s).
// Every wait is bounded; a timeout raises the status word and all roles fall through to
// the exit.
#include <cuda_bf16.h>

#include "lbp_internal.h"
#include "ptx_sm100.cuh"
#include "wht_device.cuh"
#include "wht_mma.cuh"
#include "wht_project.cuh"

namespace lbp {
namespace umma {

constexpr int kTileBytes = 64 * 128;             // 64 tokens x 64 channels of bf16
constexpr int kStageBytes = 4 * kTileBytes;      // 32 KB: an item, or a quarter of one at order 16
constexpr int kProducers = 4;
constexpr int kMaxGroups = 4;                    // epilogue warpgroups
constexpr int kThreads = (8 + 4 * kMaxGroups) * 32;
constexpr int kMaxStages = 6;
constexpr int kBarBytes = 256;
constexpr int kSmemMax = 227 * 1024;
constexpr uint32_t kTmemCols = 512;
constexpr int kSlots = 4;                        // accumulator slots (items in flight)
constexpr uint32_t kSlotCols = kTmemCols / kSlots, kHalfCols = kSlotCols / 2;

// Steps between a cursor's consecutive chunks, so that it moves without divisions.
struct Steps {
  uint32_t col, bw, bh, b;
};
struct Params {
  int32_t Hb, Wb;                // blocks (order 4: strips) of an image
  int32_t Wblocks, per_strip;    // blocks along W; blocks per cursor step along W (order 4: 4, else 1)
  int32_t r;
  int32_t C[2], cols[2];         // channels; chunks per block
  uint32_t n_chunks0, n_chunks;  // chunks of tensor 0, of both
  uint32_t* status;
  float scale[2];
  int32_t defer_wait, test_stall;
  int32_t stages, groups;        // ring stages; epilogue warpgroups at work
  Steps step[2];
};

// Chunk number -> tensor, block and column.  The position is decoded once, then
// moved by precomputed steps with carries.
struct Cursor {
  uint32_t chunk, which, col, bw, bh, b;
  __device__ __forceinline__ void decode(const Params& p, uint32_t s) {
    chunk = s;
    which = s >= p.n_chunks0 ? 1u : 0u;
    const uint32_t local = s - (which ? p.n_chunks0 : 0u);
    const uint32_t np = static_cast<uint32_t>(p.cols[which]);
    const uint32_t blk = local / np;
    col = local - blk * np;
    const uint32_t t2 = blk / p.Wb;
    bw = blk - t2 * p.Wb;
    b = t2 / p.Hb;
    bh = t2 - b * p.Hb;
  }
  __device__ __forceinline__ void advance(const Params& p, uint32_t stride) {
    const uint32_t next = chunk + stride;
    if (which == 0u && next >= p.n_chunks0) {   // into the second tensor: once per cursor
      decode(p, next);
      return;
    }
    chunk = next;
    const Steps& st = p.step[which];
    const uint32_t np = static_cast<uint32_t>(p.cols[which]);
    col += st.col;
    uint32_t carry = col >= np ? 1u : 0u;
    col -= carry ? np : 0u;
    bw += st.bw + carry;
    carry = bw >= static_cast<uint32_t>(p.Wb) ? 1u : 0u;
    bw -= carry ? p.Wb : 0u;
    bh += st.bh + carry;
    carry = bh >= static_cast<uint32_t>(p.Hb) ? 1u : 0u;
    bh -= carry ? p.Hb : 0u;
    b += st.b + carry;
  }
};

__device__ __forceinline__ void tma_store_4d_hint(const CUtensorMap* m, const void* smem_src, int32_t x,
                                                  int32_t y, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%2, %3, %4, %4}], [%1], "
      "%5;" ::"l"(reinterpret_cast<uint64_t>(m)),
      "r"(ptx::smem_u32(smem_src)), "r"(x), "r"(y), "r"(0), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// every store this thread has committed has read its source
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void group_sync(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }
__device__ __forceinline__ bool group_or(int id, bool pred) {
  uint32_t any;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %2, 0;\n\t"
      "bar.red.or.pred p, %1, 128, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(any)
      : "r"(id), "r"(static_cast<uint32_t>(pred))
      : "memory");
  return any != 0;
}

// Output maps of the tensors: boxes of the rows of a whole "block" (order 4: of the
// four blocks of a strip) and, order 4, of the last strip of a row of blocks.
struct OutMaps {
  CUtensorMap full[2], tail[2];
};

// K: order; NB: N / 16 (order 4: what the epilogue reads of a block's 16 columns, / 4)
template <int K, int NB>
__global__ void __launch_bounds__(kThreads, 1)
    wht_project_umma_kernel(const __grid_constant__ CUtensorMap tmap0,
                            const __grid_constant__ CUtensorMap tmap1,
                            const __grid_constant__ OutMaps om, const __grid_constant__ Params p,
                            const __grid_constant__ MmaPlan mp) {
  constexpr int kParts = K == 16 ? 4 : 1;
  constexpr int kN = K == 4 ? 16 : NB * 16;   // columns of one MMA
  constexpr int kPanelBytes = kN * 128;       // 64 tokens x N rows
  constexpr int kBoxH = K == 8 ? 8 : 4, kBoxW = K == 8 ? 8 : 16;   // tokens of a chunk
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sB = smem + p.stages * kStageBytes;
  uint8_t* sOut = sB + kParts * kPanelBytes;
  const int rows = p.r * p.per_strip;             // coefficient rows of a chunk
  const int out_bytes = rows * 128;
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(sOut + 4 * p.groups * out_bytes);   // [kMaxStages]
  uint64_t* empty_bar = full_bar + kMaxStages;
  uint64_t* acc_full = empty_bar + kMaxStages;   // [kSlots]
  uint64_t* acc_empty = acc_full + kSlots;       // [kSlots]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + kSlots);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // Set-up.  The loads wait for the barriers alone, which the producers' own warps set up;
  // the other warps meanwhile lay out the basis matrix and allocate TMEM (a batch of
  // 896 -> 3584 and 3584 -> 896 with 1024 tokens at order 16 48.4 -> 47.0 us, 48 -> 192 and
  // 192 -> 48 with 200704 tokens 95.8 -> 94.4).
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      ptx::mbar_init(&full_bar[s], kProducers);
      ptx::mbar_init(&empty_bar[s], 1);
    }
    for (int s = 0; s < kSlots; ++s) {
      ptx::mbar_init(&acc_full[s], 1);
      ptx::mbar_init(&acc_empty[s], 4);   // the four warps of the item's epilogue warpgroup
    }
    ptx::mbar_fence_init();
    *abort_flag = 0;
  }
  if (warp == 4) {
    ptx::tmem_alloc(tmem_slot, kTmemCols);
    ptx::tmem_relinquish();
  } else if (warp == 5 && lane < 4) {
    ptx::prefetch_tensormap(lane == 0 ? &tmap0 : lane == 1 ? &tmap1 : &om.full[lane - 2]);
  } else if (warp >= 8) {
    // The basis matrix as K-major B operands, one panel per part of 64 tokens: row n = 64
    // tokens = 128 bytes, 16-byte piece c of row n at piece c ^ (n & 7); rows past the
    // bases are zero.  Order 4 uses the first 16 tokens of a row, those of a block.
    for (int e = threadIdx.x - 256; e < kParts * kN * 8; e += kThreads - 256) {
      const int part = e / (kN * 8), n = (e >> 3) % kN, c = e & 7;
      uint32_t w[4];
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        uint32_t bits = 0u;
        const int t = c * 8 + h;
        if constexpr (K == 4) {
          if (t < 16) bits = basis_bits<4>(mp, n, p.r, t);
        } else {
          bits = basis_bits<K>(mp, n, p.r, part * 64 + t);
        }
        w[h >> 1] = (h & 1) ? w[h >> 1] | (bits << 16) : bits;
      }
      *reinterpret_cast<uint4*>(sB + part * kPanelBytes + n * 128 + ((c ^ (n & 7)) << 4)) =
          make_uint4(w[0], w[1], w[2], w[3]);
    }
    ptx::fence_proxy_async_smem();   // the tensor core reads B through the async proxy
  }
  // launched the same way behind an earlier kernel on the stream that may still
  // read the buffers written below: nothing is read or written before it has
  // completed, unless the caller vouches for disjoint buffers (then the wait
  // moves to the end and only keeps completion ordered)
  if (warp < kProducers) {
    group_sync(1 + kMaxGroups);
    asm volatile("bar.arrive %0, %1;" ::"r"(2 + kMaxGroups), "n"(kThreads) : "memory");
    if (!p.defer_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
    // A kernel launched behind this one the same way may set itself up as SMs free up; it
    // still waits for this grid before reading.  Only now: whatever starts after this
    // point may take it that the kernel ahead of this one has completed.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  } else {
    ptx::tc_fence_before_sync();
    asm volatile("bar.sync %0, %1;" ::"r"(2 + kMaxGroups), "n"(kThreads) : "memory");
    ptx::tc_fence_after_sync();
  }
  const uint32_t tmem_base = warp < kProducers ? 0u : *tmem_slot;

  // items dealt to the CTAs round robin
  const uint32_t n_items = (p.n_chunks + 3) / 4;
  const uint32_t my_items = blockIdx.x < n_items ? (n_items - blockIdx.x + gridDim.x - 1) / gridDim.x : 0u;
  const uint32_t stride = 4u * gridDim.x;   // chunks between a CTA's consecutive items

  if (warp < kProducers) {
    // =========================== TMA producers ===========================
    // One 8 KB box per chunk, each from a warp of its own: a thread issues TMA
    // requests too slowly to fetch an item alone.
    if (ptx::elect_one()) {
      // x and g_y are read exactly once: they should not push the coefficients
      // just written (read back from L2 by the next kernel) out of L2
      const uint64_t stream_once = ptx::l2_policy_evict_first();
      Cursor c;
      c.decode(p, 4 * blockIdx.x + warp);
      bool ok = true;
      int s = 0;
      uint32_t phase = 0;
      for (uint32_t n = 0; n < my_items && !p.test_stall && ok; ++n) {
        const int ch = static_cast<int>(c.col) * 64;
        const bool have = c.chunk < p.n_chunks;
        for (int part = 0; part < kParts; ++part) {
          if (!ptx::mbar_wait(&empty_bar[s], phase ^ 1u, p.status, (6u << 16) | 1u)) {
            ok = false;
            break;
          }
          if (have) {
            // the whole box counts, also where it hangs over the tensor (zero fill)
            ptx::mbar_expect_tx(&full_bar[s], kTileBytes);
            constexpr int kBoxes = K == 4 ? 4 : 1;
#pragma unroll
            for (int j = 0; j < kBoxes; ++j)
              ptx::tma_load_4d_hint(smem + s * kStageBytes + warp * kTileBytes + j * (kTileBytes / kBoxes),
                                    c.which ? &tmap1 : &tmap0, &full_bar[s], ch,
                                    static_cast<int32_t>(c.bw * kBoxW) + j * 4,
                                    static_cast<int32_t>(c.bh * (K == 16 ? 16 : kBoxH) + part * 4),
                                    static_cast<int32_t>(c.b), stream_once);
          } else {
            ptx::mbar_arrive(&full_bar[s]);   // no such chunk: what lies in the stage is multiplied and dropped
          }
          if (++s == p.stages) {
            s = 0;
            phase ^= 1u;
          }
        }
        if (ok && n + 1 < my_items) c.advance(p, stride);
      }
      if (!ok) *abort_flag = 1;
    }
  } else if (warp == 4) {
    // =========================== tcgen05 issuer ===========================
    if (ptx::elect_one()) {
      constexpr uint32_t idesc = ptx::idesc_bf16(128, kN, true, false);
      const uint32_t b_addr = ptx::smem_u32(sB);
      bool ok = true;
      int s = 0;
      uint32_t phase = 0;
      for (uint32_t n = 0; n < my_items && ok; ++n) {
        const int slot = static_cast<int>(n % kSlots);
        const bool second = 4 * (blockIdx.x + n * gridDim.x) + 2 < p.n_chunks;   // of the two halves of an item
        if (!ptx::mbar_wait(&acc_empty[slot], ((n / kSlots) + 1) & 1u, p.status, (6u << 16) | 2u)) {
          ok = false;
          break;
        }
        for (int part = 0; part < kParts; ++part) {
          if (!ptx::mbar_wait(&full_bar[s], phase, p.status, (6u << 16) | 3u)) {
            ok = false;
            break;
          }
          ptx::tc_fence_after_sync();
          const uint32_t sa = ptx::smem_u32(smem + s * kStageBytes);
          for (int h = 0; h < (second ? 2 : 1); ++h) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              // A: MN-major, 16 tokens = 16 rows of 128 bytes further per step, the two
              // chunks 8 KB apart; B: K-major, 16 tokens = 32 bytes further.  Order 4: a step
              // is a block with the one basis matrix and columns of its own.
              const uint64_t da = ptx::smem_desc_sw128(sa + h * 2 * kTileBytes + kk * 2048, kTileBytes, 1024);
              const uint64_t db =
                  ptx::smem_desc_sw128(b_addr + part * kPanelBytes + (K == 4 ? 0 : kk * 32), 16, 1024);
              ptx::mma_bf16_ss(tmem_base + slot * kSlotCols + h * kHalfCols + (K == 4 ? kk * kN : 0), da, db, idesc,
                               (K == 4 || (part == 0 && kk == 0)) ? 0u : 1u);
            }
          }
          ptx::mma_commit(&empty_bar[s]);
          if (++s == p.stages) {
            s = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        ptx::mma_commit(&acc_full[slot]);
      }
      if (!ok) *abort_flag = 1;
    }
  } else if (warp >= 8) {
    // =========================== epilogue ===========================
    // Warpgroup g takes the CTA's items g, g + groups, ...; its warps read their lane quarter.
    const int g = (warp - 8) >> 2, quarter = warp & 3;
    const bool first = quarter == 0 && lane == 0;
    const uint64_t keep = ptx::l2_policy_evict_last();   // read back from L2 by the next kernel
    uint8_t* const out = sOut + g * 4 * out_bytes;
    for (uint32_t n = g < p.groups ? g : my_items; n < my_items; n += p.groups) {
      const int slot = static_cast<int>(n % kSlots);
      const bool ok = ptx::mbar_wait(&acc_full[slot], (n / kSlots) & 1u, p.status, (6u << 16) | 4u);
      // the stores of the group's last item have read its buffer
      if (quarter == 0) bulk_wait_read();
      // one answer for the whole group (the flag may be raised between two reads of it)
      if (group_or(1 + g, !ok || *abort_flag != 0)) {
        if (first) *abort_flag = 1;
        break;
      }
      ptx::tc_fence_after_sync();
      const uint32_t chunk0 = 4 * (blockIdx.x + n * gridDim.x);
      const int chunks = p.n_chunks - chunk0 < 4u ? static_cast<int>(p.n_chunks - chunk0) : 4;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (2 * h < chunks) {
          // lanes 0-63 of the accumulator are the first chunk of the half, 64-127 the second
          const int i = 2 * h + (quarter >> 1);
          const float sc = p.scale[chunk0 + i >= p.n_chunks0 ? 1 : 0];
          uint16_t* const o = reinterpret_cast<uint16_t*>(out + i * out_bytes) + (quarter & 1) * 32 + lane;
          const uint32_t acc =
              tmem_base + (static_cast<uint32_t>(32 * quarter) << 16) + slot * kSlotCols + h * kHalfCols;
          if constexpr (K == 4) {
            constexpr int kCols = 4 * NB;   // columns read of a block
            uint16_t* oj = o;
            // (unrolled, the wide forms run out of registers)
#pragma unroll(kCols <= 8 ? 4 : 1)
            for (int j = 0; j < 4; ++j, oj += p.r * 64) {
              uint32_t v[kCols];
              if constexpr (kCols == 12) {
                uint32_t lo[8], hi[4];
                ptx::tmem_ld_xn<8>(acc + j * kN, lo);
                ptx::tmem_ld_xn<4>(acc + j * kN + 8, hi);
                ptx::tmem_ld_wait();
#pragma unroll
                for (int q = 0; q < 12; ++q) v[q] = q < 8 ? lo[q & 7] : hi[q & 3];
              } else {
                ptx::tmem_ld_xn<kCols>(acc + j * kN, v);
                ptx::tmem_ld_wait();
              }
#pragma unroll
              for (int q = 0; q < kCols; q += 2) {
                const uint32_t pk = pack_bf16x2(__uint_as_float(v[q]) * sc, __uint_as_float(v[q + 1]) * sc);
                if (q < p.r) oj[q * 64] = static_cast<uint16_t>(pk);
                if (q + 1 < p.r) oj[(q + 1) * 64] = static_cast<uint16_t>(pk >> 16);
              }
            }
          } else {
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) {
              uint32_t v[16];
              ptx::tmem_ld_xn<16>(acc + nb * 16, v);
              ptx::tmem_ld_wait();
#pragma unroll
              for (int q = 0; q < 16; q += 2) {
                const uint32_t pk = pack_bf16x2(__uint_as_float(v[q]) * sc, __uint_as_float(v[q + 1]) * sc);
                if (nb * 16 + q < rows) o[(nb * 16 + q) * 64] = static_cast<uint16_t>(pk);
                if (nb * 16 + q + 1 < rows) o[(nb * 16 + q + 1) * 64] = static_cast<uint16_t>(pk >> 16);
              }
            }
          }
        }
      }
      ptx::tc_fence_before_sync();
      ptx::fence_proxy_async_smem();   // the TMA store reads through the async proxy
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&acc_empty[slot]);   // the slot may be overwritten
      group_sync(1 + g);
      if (quarter == 0 && lane < chunks) {
        Cursor c;
        c.decode(p, chunk0 + lane);
        const long long blk = (static_cast<long long>(c.b) * p.Hb + c.bh) * p.Wblocks + c.bw * p.per_strip;
        const bool tail = K == 4 && static_cast<int>(c.bw * 4 + 4) > p.Wblocks;
        tma_store_4d_hint(tail ? &om.tail[c.which] : &om.full[c.which], out + lane * out_bytes,
                          static_cast<int32_t>(c.col) * 64, static_cast<int32_t>(blk * p.r), keep);
      }
      if (quarter == 0) bulk_commit();
    }
    if (quarter == 0) bulk_wait_all();   // this warp's stores are complete before the CTA leaves
  }

  ptx::tc_fence_before_sync();
  __syncthreads();
  if (warp == 4) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
  // deferred: this grid must not complete before the kernel ahead of it has
  if (p.defer_wait) asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace umma

// Grid size and launch attributes under the per-thread launch shape (see ProjLaunch):
// `want` CTAs at most.
static int projection_grid(uint32_t want, int sms, cudaLaunchAttribute* attr, unsigned* n_attr) {
  const ProjLaunch shape = projection_launch();
  int cap = shape.max_ctas > 0 && shape.max_ctas < sms ? shape.max_ctas : sms;
  int grid = static_cast<int>(want < static_cast<uint32_t>(cap) ? want : cap);
  unsigned n = 0;
  if (shape.programmatic) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  if (shape.whole_tpcs && grid >= 2) {
    grid &= ~1;
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = 2;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  *n_attr = n;
  return grid;
}

bool project_umma_supported(int k, int r) { return k == 4 || ((k == 8 || k == 16) && r <= 48); }

int launch_project_umma(const void* t0, void* out0, int C0, const lbp_view* view0, const void* t1,
                        void* out1, int C1, const lbp_view* view1, int B, int H, int W,
                        const BasisPlan& bp, float scale0, float scale1, int sms, uint32_t* status,
                        cudaStream_t stream) {
  using namespace umma;
  const int K = bp.k, r = bp.r;
  const int box_w = K, box_h = K == 16 ? 4 : K;
  Params p{};
  p.per_strip = K == 4 ? 4 : 1;
  p.Hb = blocks_along(H, K);
  p.Wblocks = blocks_along(W, K);
  p.Wb = (p.Wblocks + p.per_strip - 1) / p.per_strip;
  p.r = r;
  p.C[0] = C0;
  p.C[1] = t1 != nullptr ? C1 : C0;
  p.cols[0] = (C0 + 63) / 64;
  p.cols[1] = (p.C[1] + 63) / 64;
  const long long cells = static_cast<long long>(B) * p.Hb * p.Wb;
  const long long n0 = cells * p.cols[0], n1 = t1 != nullptr ? cells * p.cols[1] : 0;
  // chunk numbers, and one stride past the last, fit 32 bits; so do the rows (the caller)
  if (n0 + n1 >= (1ll << 31)) return LBP_ERR_SHAPE;
  p.n_chunks0 = static_cast<uint32_t>(n0);
  p.n_chunks = static_cast<uint32_t>(n0 + n1);
  p.status = status;
  p.scale[0] = scale0;
  p.scale[1] = scale1;
  p.defer_wait = projection_defer_wait() ? 1 : 0;
  p.test_stall = test_stall_projection() ? 1 : 0;

  MmaPlan mp;
  for (int q = 0; q < 64; ++q) {
    mp.nat_i[q] = q < r ? bp.nat_i[q] : 0;
    mp.nat_j[q] = q < r ? bp.nat_j[q] : 0;
  }
  CUtensorMap in[2];
  OutMaps om;
  const int tail_blocks = p.Wblocks % p.per_strip;
  auto maps = [&](int i, const void* t, void* out, int C, const lbp_view* view) -> int {
    if (int e = encode_box_tensor_map(&in[i], t, LBP_BF16, B, H, W, C, 64, box_w, box_h, true, view)) return e;
    // the coefficient matrix: boxes of a chunk's rows x 64 channels
    const int rows = static_cast<int>(static_cast<long long>(B) * p.Hb * p.Wblocks * r);
    if (int e = encode_box_tensor_map(&om.full[i], out, LBP_BF16, 1, 1, rows, C, 64, r * p.per_strip, 1, false))
      return e;
    om.tail[i] = om.full[i];
    if (tail_blocks > 0)
      if (int e = encode_box_tensor_map(&om.tail[i], out, LBP_BF16, 1, 1, rows, C, 64, r * tail_blocks, 1, false))
        return e;
    return LBP_OK;
  };
  if (int e = maps(0, t0, out0, C0, view0)) return e;
  if (t1 != nullptr) {
    if (int e = maps(1, t1, out1, C1, view1)) return e;
  } else {
    in[1] = in[0];
    om.full[1] = om.full[0];
    om.tail[1] = om.tail[0];
  }

  const int rows = r * p.per_strip, parts = K == 16 ? 4 : 1;
  const int nb = K == 4 ? (r + 3) / 4 : (r + 15) / 16;
  const int fixed = 1024 + kBarBytes + parts * (K == 4 ? 1 : nb) * 2048;
  auto ring = [&](int groups) { return (kSmemMax - fixed - 4 * groups * rows * 128) / kStageBytes; };
  p.groups = kMaxGroups;
  while (p.groups > 2 && ring(p.groups) < 4) --p.groups;
  p.stages = ring(p.groups) < kMaxStages ? ring(p.groups) : kMaxStages;
  const int smem_bytes = fixed + p.stages * kStageBytes + 4 * p.groups * rows * 128;

  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  // Alone on the chip the kernel is bound by HBM before it runs out of SMs: 201 MB in 43
  // us on 96 to 128 of 148 SMs and 45 on all, 77 MB of 14 x 14 or 56 x 56 grids in 24.6
  // us on 112, 22.6 on 128, 22.8 on all.  Beside a products kernel the caller's launch
  // shape says how many it gets.
  const int sms_alone = projection_launch().max_ctas > 0 ? sms : (7 * sms + 7) / 8;
  const int grid = projection_grid((p.n_chunks + 3) / 4, sms_alone, attr, &cfg.numAttrs);
  for (int w = 0; w < 2; ++w) {
    const uint32_t stride = 4u * static_cast<uint32_t>(grid), np = static_cast<uint32_t>(p.cols[w]);
    const uint32_t blk = stride / np, t2 = blk / p.Wb;
    p.step[w] = Steps{stride - blk * np, blk % p.Wb, t2 % p.Hb, t2 / p.Hb};
  }
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  auto launch = [&](auto kern, PerDevice& configured) -> int {
    if (int e = allow_dynamic_smem(configured, reinterpret_cast<const void*>(kern), kSmemMax)) return e;
    LBP_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, in[0], in[1], om, p, mp));
    count_launch();
    return LBP_OK;
  };
  static PerDevice configured[3][4];
#define LBP_CASE(KK, NB) \
  case KK * 10 + NB: return launch(wht_project_umma_kernel<KK, NB>, configured[KK / 8][NB - 1])
  switch (K * 10 + nb) {
    LBP_CASE(4, 1);
    LBP_CASE(4, 2);
    LBP_CASE(4, 3);
    LBP_CASE(4, 4);
    LBP_CASE(8, 1);
    LBP_CASE(8, 2);
    LBP_CASE(8, 3);
    LBP_CASE(16, 1);
    LBP_CASE(16, 2);
    LBP_CASE(16, 3);
  }
#undef LBP_CASE
  return LBP_ERR_BASIS;
}

}  // namespace lbp
