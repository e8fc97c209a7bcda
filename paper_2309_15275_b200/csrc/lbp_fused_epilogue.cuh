// Epilogue of one accumulator tile of the products kernel: a GW tile is written
// to g_W (or to an fp32 K-slice plane); a GX tile is expanded with the transposed
// bases (Eq. 7) and written to g_x, so g_x_hat never leaves the chip.
//
// Eight warps form a group, two per TMEM lane quarter: two halves of four warps that
// take different blocks (GX) or columns (GW) of a tile.  Sixteen warps in all: the
// chain of one block (accumulator read, butterfly, shared stores, hand-over) is bound
// by latency, a warp alone issues an instruction every four to five cycles.
//
// GX: the accumulator holds g_x_hat transposed, one channel per TMEM lane and one
// low-rank row per column, so a thread reads all coefficients of a block for its
// channel with tcgen05.ld and needs no other thread's data: butterfly in
// registers, one bf16 per distinct token value into a shared-memory tile of
// T x T tokens x 128 channels, and TMA stores from there, issued by a warp of their own
// (one per group), so that the eight warps never wait for one another.  A Walsh row
// of sequency below LB is constant on runs of K / LB tokens; the repetition over
// tokens is left to the TMA: the tile is stored S x S times, each time through a
// tensor map that addresses every S-th token (S = K / T), which writes each distinct
// value to shared memory once instead of S * S times and clips what hangs over the
// grid.  What bounds it: an SM's stores.  TMA stores of 256-byte rows move 51 GB/s
// from one SM and 5.3-5.8 TB/s from all (128-byte rows: 26 and 3.5; a warp's 8-byte
// stores to four 64-byte pieces, the earlier form of this epilogue, 34 and 4.3).
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "lbp_fused.cuh"
#include "ptx_sm100.cuh"
#include "wht_device.cuh"

namespace lbp {
namespace fused {

constexpr int BM = 128;
constexpr int kEGroups = 2;            // epilogue groups of 8 warps
constexpr int kGroupBytes = 32768;     // a group's buffers
constexpr int kGwStageBytes = BM * 32 * 4;   // a 32-column chunk of a GW tile
constexpr int kStoreMapsMax = 16;

// Forms of the expansion (template CORE): 2, 4: a 2 x 2 / 4 x 4 array of
// coefficients.  8: an 8 x 8 array as four 4 x 4 quadrants: with u = 2 a + d, v = 2 b
// + e, natural row index 2 m + h, the Walsh sign factors into that of (m, a) and
// (-1)^(h d), and h = 1 exactly where the sequency is 4 or more, so
//   value(u, v) = Q00[a][b] + (-1)^d Q10[a][b] + (-1)^e Q01[a][b] + (-1)^(d+e) Q11[a][b]
// with Qhh' the 4 x 4 transform of a quadrant.  7: the same with Q11 empty (every
// LP_L1 set of the paper).  6: also at most one basis in Q10 and one in Q01 (PREFIX
// sets of rank 14-16): their quadrants are a sign times one coefficient, and an 8 x 8
// block costs 160 additions instead of 384.
constexpr int kCoreSparse = 6, kCoreNoHH = 7;

template <int K, int CORE>
struct Expand {
  static constexpr int LB = CORE > 4 ? 8 : CORE;
  static constexpr int T = LB <= 4 ? 4 : 8;   // side of the stored tile
  static constexpr int S = K / T;             // token stride of a store
  static constexpr int kMaps = S * S;
  // A fill is what a group hands to the TMA at a time: of two blocks, one from either
  // half, four token rows each (a hand-over costs a warp about 200 cycles: with two
  // rows of an 8 x 8 tile at a time half of the expansion's time).
  static constexpr int kHalfBytes = 4 * T * 256;
  static constexpr int kFillBytes = 2 * kHalfBytes;
  static constexpr int kBoxRows = kHalfBytes / (T * 256);   // token rows of one store
  static constexpr int kParts = T / kBoxRows;               // fills per two blocks
  static constexpr int kBufs = kGroupBytes / kFillBytes;
  static_assert(2 * kGwStageBytes <= kGroupBytes, "a GW chunk of either half fits the group's buffers");
  static_assert(K % T == 0 && kMaps <= kStoreMapsMax, "store geometry");
};

struct StoreMaps {
  CUtensorMap m[kStoreMapsMax];
  CUtensorMap extra;   // g_x of the tokens outside the grid: boxes of 32 tokens x 128 channels
};

__device__ __forceinline__ void named_bar_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Barrier over `nthreads` threads that also ORs a predicate over them: every
// participant gets the same answer, so a decision taken on it (leave the tile
// loop after an expired wait) cannot split the threads that share the barrier.
__device__ __forceinline__ bool named_bar_or(int id, int nthreads, bool pred) {
  uint32_t any;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %3, 0;\n\t"
      "bar.red.or.pred p, %1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(any)
      : "r"(id), "r"(nthreads), "r"(static_cast<uint32_t>(pred))
      : "memory");
  return any != 0;
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* m, const void* smem_src, int32_t c0,
                                             int32_t c1, int32_t c2, int32_t c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
          reinterpret_cast<uint64_t>(m)),
      "r"(ptx::smem_u32(smem_src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// at most N of this thread's latest store groups have not yet read their source
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// What the epilogue needs to know about the accumulator it drains.
struct DrainTile {
  int row_base;       // GW: first g_W row of these 128 accumulator rows; GX: first channel of the 128 lanes
  int row_tile;       // GX: row tile
  int col_base;       // GW: first g_W column
  int slice;          // GW: K slice (plane index when gw_splits > 1)
  uint32_t tmem_acc;  // TMEM address of column 0, lane 0 of the accumulator
};

// A warp has read its last accumulator column of the tile.
template <class Release>
__device__ __forceinline__ void release_slot(int lane, Release release) {
  ptx::tc_fence_before_sync();
  __syncwarp();
  if (lane == 0) release();
}

// ---- GW tile: g_W[row_base + row, col_base + col] ----
// Every half takes the 32-column chunks half, half + 4, ... on its own: a chunk is
// staged in shared memory and written out with eight lanes along a row, so that a
// store instruction covers whole 128-byte pieces of four rows.
template <class Release>
__device__ __forceinline__ void drain_gw(const FusedParams& p, const DrainTile& t, float* E, int bar_id,
                                         int half, int quarter, int lane, Release release) {
  constexpr int kHalves = 2 * kEGroups;
  constexpr int kStride = 32;   // fp32 words per staged row; 16-byte piece c of row i sits at piece c ^ (i & 7)
  const uint32_t lane_bits = static_cast<uint32_t>(quarter * 32) << 16;
  const int ew = quarter;
  const bool planes = p.gw_splits > 1;
  bool released = false;
  for (int c0 = half * 32; c0 < p.BNw; c0 += 32 * kHalves) {
    uint32_t v[32];
    ptx::tmem_ld_32x32(t.tmem_acc + lane_bits + c0, v);
    ptx::tmem_ld_wait();
    if (c0 + 32 * kHalves >= p.BNw) {
      released = true;
      release_slot(lane, release);
    }
    const int erow_i = quarter * 32 + lane;
    uint4* erow = reinterpret_cast<uint4*>(E + erow_i * kStride);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      erow[q ^ (erow_i & 7)] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    named_bar_sync(bar_id, 128);
    if (planes || !p.gw_bf16) {
      // fp32 g_W, or a K slice: fp32 partial plane, summed by the reduce kernel that follows
      float* dst = planes ? p.gw_planes + static_cast<long long>(t.slice) * p.Cout * p.Cin
                          : static_cast<float*>(p.g_W);
      const bool add = !planes && p.beta != 0.f;
      const int o = lane & 7, rs = lane >> 3;
      const int col = t.col_base + c0 + o * 4;
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        const int row = it * 16 + ew * 4 + rs;
        const long long grow = static_cast<long long>(t.row_base) + row;
        if (grow < p.Cout && col < p.Cin) {
          float4 f = *reinterpret_cast<const float4*>(E + row * kStride + ((o ^ (row & 7)) << 2));
          float4* at = reinterpret_cast<float4*>(dst + grow * p.Cin + col);
          if (add) {
            const float4 old = *at;
            f.x = fmaf(p.beta, old.x, f.x);
            f.y = fmaf(p.beta, old.y, f.y);
            f.z = fmaf(p.beta, old.z, f.z);
            f.w = fmaf(p.beta, old.w, f.w);
          }
          *at = f;
        }
      }
    } else {
      __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(p.g_W);
      const int o = lane & 3, rs = lane >> 2;
      const int col = t.col_base + c0 + o * 8;
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        const int row = it * 32 + ew * 8 + rs;
        const long long grow = static_cast<long long>(t.row_base) + row;
        if (grow < p.Cout && col < p.Cin) {
          float4 f0 =
              *reinterpret_cast<const float4*>(E + row * kStride + (((2 * o) ^ (row & 7)) << 2));
          float4 f1 =
              *reinterpret_cast<const float4*>(E + row * kStride + (((2 * o + 1) ^ (row & 7)) << 2));
          uint4* at = reinterpret_cast<uint4*>(dst + grow * p.Cin + col);
          if (p.beta != 0.f) {
            const uint4 old = *at;
            f0.x = fmaf(p.beta, bf16_lo(old.x), f0.x);
            f0.y = fmaf(p.beta, bf16_hi(old.x), f0.y);
            f0.z = fmaf(p.beta, bf16_lo(old.y), f0.z);
            f0.w = fmaf(p.beta, bf16_hi(old.y), f0.w);
            f1.x = fmaf(p.beta, bf16_lo(old.z), f1.x);
            f1.y = fmaf(p.beta, bf16_hi(old.z), f1.y);
            f1.z = fmaf(p.beta, bf16_lo(old.w), f1.z);
            f1.w = fmaf(p.beta, bf16_hi(old.w), f1.w);
          }
          *at = make_uint4(pack_bf16x2(f0.x, f0.y), pack_bf16x2(f0.z, f0.w), pack_bf16x2(f1.x, f1.y),
                           pack_bf16x2(f1.z, f1.w));
        }
      }
    }
    named_bar_sync(bar_id, 128);
  }
  if (!released) release_slot(lane, release);   // this half had no chunk of the tile
}

// A group's buffers on their way from the epilogue warps to the warp that issues
// their TMA stores.  `count` runs over all fills of the group; fill n lies in buffer
// n % kBufs.  full[b]: the eight warps have written it; empty[b]: its stores have read it.
template <class X>
struct Fills {
  static constexpr int BUFS = X::kBufs;
  static constexpr int kInFlight = BUFS / 2;   // fills the store warp leaves in flight behind it
  uint8_t* buf;
  uint64_t* full;    // [BUFS]
  uint64_t* empty;   // [BUFS]
  uint32_t* status;
  uint32_t count;
  uint32_t returned;   // store warp: buffers given back
  __device__ __forceinline__ uint8_t* at(uint32_t n) const { return buf + (n % BUFS) * X::kFillBytes; }
  // writers: the buffer of fill n may be written
  __device__ __forceinline__ bool wait_empty(uint32_t n) const {
    return ptx::mbar_wait(&empty[n % BUFS], ((n / BUFS) + 1) & 1u, status, (5u << 16) | 6u);
  }
  // writers: this warp's part of fill `count` is written
  __device__ __forceinline__ void written(int lane) {
    ptx::fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(&full[count % BUFS]);
    ++count;
  }
  // store warp: fill `count` has been issued; give back what no longer can be read
  __device__ __forceinline__ void issued(int lane) {
    bulk_commit();
    ++count;
    bulk_wait_read<kInFlight>();
    __syncwarp();
    if (count - returned > kInFlight) {
      if (lane == 0) ptx::mbar_arrive(&empty[returned % BUFS]);
      ++returned;
    }
  }
  // store warp: wait for all stores and give every buffer back
  __device__ __forceinline__ void flush(int lane) {
    bulk_wait_read<0>();
    __syncwarp();
    for (; returned != count; ++returned)
      if (lane == 0) ptx::mbar_arrive(&empty[returned % BUFS]);
  }
};

// ---- GX tile of tokens outside the grid: g_x[token, channel], no expansion ----
// The drains of GX tiles return false when a wait expired.
template <class F, class Release>
__device__ __forceinline__ bool drain_gx_extra(const FusedParams& p, const DrainTile& t, F& fills, int eg,
                                               int sub, int quarter, int lane, Release release) {
  const uint32_t lane_bits = static_cast<uint32_t>(quarter * 32) << 16;
  bool released = false;
  constexpr int kRowBytes = 256;
  for (int c0 = eg * 32; c0 < p.BNx; c0 += 32 * kEGroups) {
    uint32_t v[16];   // 16 tokens
    ptx::tmem_ld_32x16(t.tmem_acc + lane_bits + c0 + sub * 16, v);
    ptx::tmem_ld_wait();
    if (c0 + 32 * kEGroups >= p.BNx) {
      released = true;
      release_slot(lane, release);
    }
    if (!__all_sync(0xffffffffu, fills.wait_empty(fills.count))) return false;
    uint16_t* const o =
        reinterpret_cast<uint16_t*>(fills.at(fills.count) + sub * 16 * kRowBytes) + quarter * 32 + lane;
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
      const uint32_t pk = pack_bf16x2(__uint_as_float(v[j]), __uint_as_float(v[j + 1]));
      o[j * 128] = static_cast<uint16_t>(pk);
      o[(j + 1) * 128] = static_cast<uint16_t>(pk >> 16);
    }
    fills.written(lane);
  }
  if (!released) release_slot(lane, release);
  return true;
}

// Natural (Sylvester) row index of sequency s at order n: the bits of the Gray code
// of s, reversed.
__host__ __device__ constexpr int nat_index(int n, int s) {
  const int gray = s ^ (s >> 1);
  int r = 0;
  for (int bit = 1, rev = n >> 1; bit < n; bit <<= 1, rev >>= 1)
    if (gray & bit) r |= rev;
  return r;
}

// N x N coefficients of a block (positions pos0 ..) from the accumulator columns at `at`,
// one load each.  Unselected positions read column 0 of the block and drop it
// (mask_transform): a branch around a tcgen05.ld costs more than the load.
template <int N>
__device__ __forceinline__ void read_coeffs(uint32_t at, const FusedBasis& fb, int pos0,
                                            float (&q)[N][N][1]) {
#pragma unroll
  for (int a = 0; a < N; ++a)
#pragma unroll
    for (int b = 0; b < N; ++b)
      q[a][b][0] = __uint_as_float(ptx::tmem_ld_x1(at + fb.col[pos0 + a * N + b]));
}
// The same where the slots are ordered by rows: one load of N columns per row (27
// cycles a load in these kernels, whatever its width).  What it reads past a row's
// end is masked like any unselected position.
template <int N>
__device__ __forceinline__ void read_rows(uint32_t at, const FusedBasis& fb, float (&q)[N][N][1]) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    uint32_t v[N];
    ptx::tmem_ld_xn<N>(at + fb.row[i], v);
#pragma unroll
    for (int j = 0; j < N; ++j) q[nat_index(N, i)][nat_index(N, j)][0] = __uint_as_float(v[j]);
  }
}
// A wide load of a block at TMEM column c may reach this far past its r columns.
__device__ __forceinline__ bool rows_fit(const FusedBasis& fb, uint32_t taddr, int r, int width) {
  return fb.by_rows != 0 && static_cast<int>(taddr & 0xffffu) + r + width <= 512;
}
template <int N>
__device__ __forceinline__ void mask_transform(const FusedBasis& fb, int pos0, float scale,
                                               float (&q)[N][N][1]) {
#pragma unroll
  for (int a = 0; a < N; ++a)
#pragma unroll
    for (int b = 0; b < N; ++b)
      q[a][b][0] = __uint_as_float(__float_as_uint(q[a][b][0]) & fb.keep[pos0 + a * N + b]);
  if (scale != 1.f) {
#pragma unroll
    for (int a = 0; a < N; ++a)
#pragma unroll
      for (int b = 0; b < N; ++b) q[a][b][0] *= scale;
  }
  hadamard_rows<N, 1>(q);
  hadamard_cols<N, 1>(q);
}

// ---- GX tile: expand g_x_hat (128 channels x BNx low-rank rows) into g_x ----
template <int K, int CORE, class F, class Release>
__device__ __forceinline__ bool drain_gx(const FusedParams& p, const FusedBasis& fb, const DrainTile& t,
                                         F& fills, int eg, int sub, int quarter, int lane,
                                         Release release) {
  using X = Expand<K, CORE>;
  const uint32_t acc0 = t.tmem_acc + (static_cast<uint32_t>(quarter * 32) << 16);
  const int blk0 = t.row_tile * p.bpt;
  const int n_blocks = p.nb - blk0 < p.bpt ? p.nb - blk0 : p.bpt;
  const bool live = t.row_base + quarter * 32 < p.Cin;   // some of this warp's channels exist
  bool released = false;
  // a fill takes two blocks, one of either half; the last one may have a block of the
  // first half only: the other half then reads it too and writes nothing
  for (int j0 = 2 * eg; j0 < n_blocks; j0 += 2 * kEGroups) {
    const bool mine = live && j0 + sub < n_blocks;
    const uint32_t at = acc0 + (j0 + sub < n_blocks ? j0 + sub : j0) * p.r;
    auto release_if_last = [&]() {
      if (j0 + 2 * kEGroups >= n_blocks) {
        released = true;
        release_slot(lane, release);
      }
    };
    if constexpr (X::LB <= 4) {
      constexpr int LB = X::LB, REP = X::T / LB;
      float q[LB][LB][1];
      if (rows_fit(fb, at, p.r, LB))
        read_rows<LB>(at, fb, q);
      else
        read_coeffs<LB>(at, fb, 0, q);
      ptx::tmem_ld_wait();
      release_if_last();
      mask_transform<LB>(fb, 0, p.gx_scale, q);
      if (!__all_sync(0xffffffffu, fills.wait_empty(fills.count))) return false;
      if (mine) {
        uint16_t* const o =
            reinterpret_cast<uint16_t*>(fills.at(fills.count) + sub * X::kHalfBytes) + quarter * 32 + lane;
#pragma unroll
        for (int u = 0; u < X::T; ++u)
#pragma unroll
          for (int b = 0; b < LB; b += 2) {
            const uint32_t pk = pack_bf16x2(q[u / REP][b][0], q[u / REP][b + 1][0]);
#pragma unroll
            for (int d = 0; d < REP; ++d) {
              o[(u * X::T + b * REP + d) * 128] = static_cast<uint16_t>(pk);
              o[(u * X::T + (b + 1) * REP + d) * 128] = static_cast<uint16_t>(pk >> 16);
            }
          }
      }
      fills.written(lane);
    } else {
      float q00[4][4][1], q10[4][4][1], q01[4][4][1], q11[4][4][1];
      if constexpr (CORE == kCoreSparse) {
        if (rows_fit(fb, at, p.r, 4))
          read_rows<4>(at, fb, q00);
        else
          read_coeffs<4>(at, fb, 0, q00);
        q10[0][0][0] = __uint_as_float(ptx::tmem_ld_x1(at + fb.ex_col[0]));
        q01[0][0][0] = __uint_as_float(ptx::tmem_ld_x1(at + fb.ex_col[1]));
      } else if (rows_fit(fb, at, p.r, 8)) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          uint32_t v[8];
          ptx::tmem_ld_xn<8>(at + fb.row[i], v);
          const int a = nat_index(8, i) >> 1;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int b = nat_index(8, j) >> 1;
            const float f = __uint_as_float(v[j]);
            if (i < 4 && j < 4) q00[a][b][0] = f;
            if (i >= 4 && j < 4) q10[a][b][0] = f;
            if (i < 4 && j >= 4) q01[a][b][0] = f;
            if (CORE == 8 && i >= 4 && j >= 4) q11[a][b][0] = f;
          }
        }
      } else {
        read_coeffs<4>(at, fb, 0, q00);
        read_coeffs<4>(at, fb, 16, q10);
        read_coeffs<4>(at, fb, 32, q01);
        if constexpr (CORE == 8) read_coeffs<4>(at, fb, 48, q11);
      }
      ptx::tmem_ld_wait();
      release_if_last();
      mask_transform<4>(fb, 0, p.gx_scale, q00);
      float e0 = 0.f, e1 = 0.f;
      if constexpr (CORE == kCoreSparse) {
        e0 = __uint_as_float(__float_as_uint(q10[0][0][0] * p.gx_scale) & fb.ex_keep[0]);
        e1 = __uint_as_float(__float_as_uint(q01[0][0][0] * p.gx_scale) & fb.ex_keep[1]);
      } else {
        mask_transform<4>(fb, 16, p.gx_scale, q10);
        mask_transform<4>(fb, 32, p.gx_scale, q01);
        if constexpr (CORE == 8) mask_transform<4>(fb, 48, p.gx_scale, q11);
      }
#pragma unroll
      for (int part = 0; part < X::kParts; ++part) {   // token rows 4 part ...
        if (!__all_sync(0xffffffffu, fills.wait_empty(fills.count))) return false;
        if (mine) {
          uint16_t* const o0 =
              reinterpret_cast<uint16_t*>(fills.at(fills.count) + sub * X::kHalfBytes) + quarter * 32 + lane;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int a = 2 * part + (i >> 2), b = i & 3;
            uint16_t* const o = o0 + (i >> 2) * 16 * 128;
            const float q = q00[a][b][0];
            float v00, v01, v10, v11;   // tokens (2 a + d, 2 b + e)
            if constexpr (CORE == kCoreSparse) {
              const float s0 = fb.ex_sign[0][a * 4 + b], s1 = fb.ex_sign[1][a * 4 + b];   // +-1: exact products
              const float sp = fmaf(s0, e0, q), sm = fmaf(-s0, e0, q);
              v00 = fmaf(s1, e1, sp);
              v01 = fmaf(-s1, e1, sp);
              v10 = fmaf(s1, e1, sm);
              v11 = fmaf(-s1, e1, sm);
            } else {
              const float sp = q + q10[a][b][0], sm = q - q10[a][b][0];
              float tp = q01[a][b][0], tm = q01[a][b][0];
              if constexpr (CORE == 8) {
                tp += q11[a][b][0];
                tm -= q11[a][b][0];
              }
              v00 = sp + tp;
              v01 = sp - tp;
              v10 = sm + tm;
              v11 = sm - tm;
            }
            const uint32_t row0 = pack_bf16x2(v00, v01), row1 = pack_bf16x2(v10, v11);
            o[(2 * b) * 128] = static_cast<uint16_t>(row0);
            o[(2 * b + 1) * 128] = static_cast<uint16_t>(row0 >> 16);
            o[(8 + 2 * b) * 128] = static_cast<uint16_t>(row1);
            o[(9 + 2 * b) * 128] = static_cast<uint16_t>(row1 >> 16);
          }
        }
        fills.written(lane);
      }
    }
  }
  if (!released) release_slot(lane, release);   // this group had no block of the tile
  return true;
}

// ---- the store warp of a group: the TMA stores of a GX tile's fills ----
// A lane issues one store of a fill (two blocks x kMaps) and waits for its own.
template <int K, int CORE, class F>
__device__ __forceinline__ bool store_gx(const FusedParams& p, const StoreMaps& maps, const DrainTile& t,
                                         F& fills, int eg, int lane) {
  using X = Expand<K, CORE>;
  static_assert(2 * X::kMaps <= 32, "one store per lane");
  const bool extra = t.row_tile >= p.n_rt;
  const int blk0 = t.row_tile * p.bpt;
  const int n_blocks = p.nb - blk0 < p.bpt ? p.nb - blk0 : p.bpt;
  const int first = extra ? eg * 32 : eg * 2, step = extra ? 32 * kEGroups : 2 * kEGroups;
  const int end = extra ? p.BNx : n_blocks, parts = extra ? 1 : X::kParts;
  const int j = lane / X::kMaps, m = lane % X::kMaps;
  for (int i = first; i < end; i += step) {
    // the box starts at token (y, x) of image b; boxes that hang over the grid are
    // clipped, those that lie outside are not issued
    const int blk = blk0 + i + j;
    const int bw = blk % p.Wb, t2 = blk / p.Wb, bh = t2 % p.Hb, b = t2 / p.Hb;
    for (int part = 0; part < parts; ++part) {
      const uint32_t n = fills.count;
      if (!__all_sync(0xffffffffu, ptx::mbar_wait(&fills.full[n % X::kBufs], (n / X::kBufs) & 1u,
                                                  p.status, (5u << 16) | 7u)))
        return false;
      const uint8_t* src = fills.at(n);
      if (extra) {
        const int row = (t.row_tile - p.n_rt) * p.BNx + i;
        if (lane == 0 && t.row_base < p.Cin && row < p.n_extra)
          tma_store_4d(&maps.extra, src, t.row_base, row, 0, 0);
      } else {
        const int y = bh * K + part * X::kBoxRows * X::S + m / X::S, x = bw * K + m % X::S;
        if (j < 2 && i + j < n_blocks && t.row_base < p.Cin && y < p.H && x < p.W)
          tma_store_4d(&maps.m[m], src + j * X::kHalfBytes, t.row_base, bw * X::T,
                       bh * X::T + part * X::kBoxRows, b);
      }
      fills.issued(lane);
    }
  }
  return true;
}

}  // namespace fused
}  // namespace lbp
