// fp32 products on the tcgen05 tensor cores, by splitting every operand into three bf16 parts.
//
//   D(l, c) = sum_k L(k, l) * C(k, c)
//
// L, stored (K, lanes) row-major, becomes the A operand, a TMEM lane per l; C, stored (K,
// columns) or (columns, K) row-major, the B operand.  g_W = g_y_hat^T x_hat is this with L =
// g_y_hat and C = x_hat, g_x_hat = g_y_hat W with L = W and C = g_y_hat (D transposed).
//
// x = hi + mid + lo, each part the bf16 nearest to what the parts before it leave: 8
// significant bits a part and a sign each, so the three hold x to 2^-27 of itself.  mid and lo
// are held times 2^15, which keeps them clear of the end of bf16's range (2^-133) for every
// normal x: held as they are, they lose bits of numbers below 2^-110 (g_y of 2^-114: error
// 5.7e-7, of 2^-120: 3.6e-5; now 0.9e-7 throughout).  The scaling makes a block 1 % longer.  Of
// the nine products of parts the six largest are formed; the rest is below 2^-26 of a term.
// A product of two bf16 numbers is exact in fp32, so what is left is the summation.  The
// tensor core drops bits of the smaller addend when it adds to an accumulator, so a
// k-block of 64 starts from an accumulator of its own, its small products go first, and the
// sums of k-blocks are added up in registers, rounding to nearest.
//
// An item is a tile of 128 lanes x BN columns over a run of k-blocks of 64.  TMA brings a block's
// fp32 operands to shared memory, two blocks ahead.  Of a CTA's 16 warps eight split L (a
// thread the k's of its lane) and write the parts to TMEM, the others split C and store the
// parts to shared memory in the 128-byte-swizzled layout the tensor core reads.  One thread
// of a warp of its own issues the 24 MMAs of 128 x BN x 16; under them all warps add the
// accumulator of the block before to their sums.  Two stages of everything.
//
// A 128 x 128 x 64 block takes 1.3 us (128 x 64 x 64: 1.04): its MMAs 0.8, splitting 0.7
// (conversions and shifts at half rate), one partly under the other; an item's start and end,
// with the launch, another 7 (5.6): 8.3, 9.4, 12.2, 22.4 and 37.7 us for one of 1, 2, 4, 12 and 24
// blocks alone on the chip and from cold caches (7.0, 7.5, 9.2, 17.4 and 30.0).  Tried before:
// loads into registers, issued as these become free, make every use wait for the latest load
// (2.1 us a block, from 8 or 16 warps, also with persistent CTAs, two CTAs to an SM or the parts
// of L in TMEM).  64 blocks of 448 -> 1792 at rank 10: both products 55 us on FFMA
// (37 TFLOP/s), 20.6 here (100, six times that in bf16); error against 64 bits of g_x and g_W
// 2.4e-7 and 2.5e-7 there, 1.3e-7 and 1.4e-7 here.
//
// An item of one to five k's is summed by FMAs instead: these round once per term, which is
// less than the tensor core drops from six products (relative error at 1, 2, 3, 4, 5, 6 and 8
// terms: FMAs 2.5, 3.1, 3.6, 4.0, 4.4, 4.7 and 5.4e-8, split 4.5 to 4.7e-8 at all of them).
//
// Infinities, NaN and values next to the largest float leave the parts meaningless
// (inf - inf, 0 * inf), and the scaled products of terms of 2^113 and more overflow, but all
// that always shows as a sum that is not finite; and where a sum is next to subnormal the
// tensor core's cut at 2^-149 shows, where FMAs round (g_y of 2^-130, W of 1: 1.4e-6 against
// 5.6e-7).  A CTA that has a sum not finite or below 2^-120 fetches the item's operands once more
// and its warps form their sums from them with fp32 FMAs, term by term; only such sums are
// replaced.  640 x 448 -> 1792, both products: 22 us, with one NaN in g_y 120, with nothing but
// NaN 141 (FFMA kernel 60 whatever the values; a serial sum per thread from global memory 980
// and 1120); 2048 x 768 -> 3072: 115, 250 and 803 (436; 1690 and 6850).
#include "gemm_fp32.cuh"
#include "lbp_internal.h"
#include "ptx_sm100.cuh"
#include "wht_device.cuh"

namespace lbp {
namespace split {

constexpr int kLanes = 128, kBK = 64;
constexpr int kWarps = 16;                       // 8 for L, 8 for C
constexpr int kThreads = (kWarps + 1) * 32;      // and one that issues loads and MMAs
constexpr int kShift = 15;                       // mid and lo are held times 2^15
constexpr int kFewTerms = 5;                     // an item of no more k's is left to FMAs
constexpr int kChunkBytes = 64 * kBK * 2;        // 64 columns of an MN-major operand
constexpr uint32_t kTmemCols = 512, kTmemL = 256, kPartCols = kBK / 2;   // L: two stages of three parts behind the accumulators

template <int BN>
struct Cfg {
  static constexpr int kPart = BN * kBK * 2;                  // of C
  static constexpr int kStage = 3 * kPart;
  static constexpr int kRawL = kLanes * kBK * 4, kRaw = kRawL + BN * kBK * 4;   // as TMA brings them
  static constexpr int kOut = 16 * 32 * (BN / 4) * 4;         // the sums on their way out
  static constexpr int kSmem = 2 * (kStage + kRaw) + 1024 + 64;
  static_assert(kOut <= 2 * kStage && kSmem <= 227 * 1024, "shared memory");
  static constexpr int kPieces = BN * kBK / 4 / 256;          // of four numbers, per thread
  static constexpr int kCols = BN / 4;                        // accumulator columns of a warp
};

struct Maps {
  CUtensorMap l[2], c[2];   // of either job
};

__device__ __forceinline__ void tmem_st_x8(uint32_t taddr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem desc]
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D = 2^-kShift D + A * B
__device__ __forceinline__ void mma_bf16_ts_down(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.eq.b32 p, 0, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p, %4;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "n"(kShift)
      : "memory");
}

// Both times 2^kShift, in one packed multiply (in two, a block of 128 x 128 x 64 takes 1 % longer).
__device__ __forceinline__ void scale_up(float& a, float& b) {
  asm("{\n\t.reg .b64 x, s;\n\t"
      "mov.b64 x, {%0, %1};\n\tmov.b64 s, {%2, %2};\n\t"
      "mul.rn.f32x2 x, x, s;\n\t"
      "mov.b64 {%0, %1}, x;\n\t}"
      : "+f"(a), "+f"(b)
      : "f"(static_cast<float>(1 << kShift)));
}
// The next part of two numbers (0 hi, 1 mid, 2 lo); what it leaves of them.
__device__ __forceinline__ uint32_t take_part(float& a, float& b, int part) {
  const uint32_t w = pack_bf16x2(a, b);
  a -= bf16_lo(w);   // exact
  b -= bf16_hi(w);
  if (part == 0) scale_up(a, b);
  return w;
}

// The item of this CTA.
template <int BN>
struct Item {
  const CUtensorMap *map_l, *map_c;
  uint8_t *smem, *raw;
  uint64_t* full;        // [2]: a block's operands have arrived
  uint32_t* status;
  float* D;
  long long lanes, cols, K;
  int32_t l0, c0, kb0, n_kb;
  bool wt;               // L = B, C = A stored (columns, K), D transposed

  __device__ __forceinline__ Item(const GemmFp32Jobs& jobs, const Maps& maps) {
    extern __shared__ uint8_t smem_raw[];
    smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    raw = smem + 2 * Cfg<BN>::kStage;
    full = reinterpret_cast<uint64_t*>(raw + 2 * Cfg<BN>::kRaw);
    status = jobs.status;
    int t = blockIdx.x;
    const int which = t >= jobs.items0 ? 1 : 0;
    const GemmFp32Job& g = jobs.j[which];
    map_l = &maps.l[which];
    map_c = &maps.c[which];
    if (which) t -= jobs.items0;
    const int chunk = t % g.chunks;
    t /= g.chunks;
    wt = g.a_mn == 0;
    lanes = wt ? g.N : g.M;
    cols = wt ? g.M : g.N;
    K = g.K;
    l0 = (t / g.tiles_c) * kLanes;   // (coordinates of a tensor map: below 2^31)
    c0 = (t % g.tiles_c) * BN;
    kb0 = chunk * g.per;
    n_kb = (kb0 + g.per < g.kb ? kb0 + g.per : g.kb) - kb0;
    D = g.D + chunk * g.M * g.N;
  }

  // One thread: the u-th load of this CTA, block u of the item (and u - n_kb once more from there on).
  __device__ __forceinline__ void load(int u) const {
    using C = Cfg<BN>;
    uint8_t* const dst = raw + (u & 1) * C::kRaw;
    const int k = (kb0 + (u < n_kb ? u : u - n_kb)) * kBK;
    ptx::mbar_expect_tx(&full[u & 1], C::kRaw);   // boxes count in full, also where they hang over an edge (zeros)
    ptx::tma_load_2d(dst, map_l, &full[u & 1], l0, k);
    ptx::tma_load_2d(dst + C::kRawL, map_c, &full[u & 1], wt ? k : c0, wt ? c0 : k);
  }
  __device__ __forceinline__ bool arrived(int u, uint32_t site) const {
    return ptx::mbar_wait(&full[u & 1], static_cast<uint32_t>(u >> 1) & 1u, status, (7u << 16) | site);
  }
};

// A sum that stays: zero, or a finite one of 2^-120 and more.
constexpr float kLeastSum = 0x1p-120f, kMostSum = 3.402823466e38f;
__device__ __forceinline__ bool stays(float v) {
  return v == 0.f || (fabsf(v) >= kLeastSum && fabsf(v) <= kMostSum);
}

// The rest of an item by FMAs, with all threads of the CTA: its sums term by term, one k after
// the other.  few: its only block has been fetched.  Otherwise the item is fetched once more,
// and of the sums in smem = [kCols][threads] those that do not stay are replaced, in warps with
// `mine` set.  A thread has kCols / 4 lanes (in runs of four) by 4 columns, which reads less
// than a lane by kCols.  Not inlined, and with nothing handed over: registers that the kernel
// spills for this path cost every item of one block 0.5 us.
template <int BN>
__device__ __noinline__ void finish_by_fma(const GemmFp32Jobs& jobs, const Maps& maps, bool few, bool mine) {
  using C = Cfg<BN>;
  const Item<BN> item(jobs, maps);
  const float* const old = reinterpret_cast<const float*>(item.smem);
  constexpr int kRuns = C::kCols / 16, kAlong = 8 / kRuns;   // runs of a thread; threads along the lanes
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int run = (lane % kAlong) * 4, four = lane / kAlong * 4;
  const bool wt = item.wt;
  const int l_at = (warp & 3) * 32 + run, c_at = C::kRawL / 4 + ((warp >> 2) * C::kCols + four) * (wt ? kBK : 1);
  float sum[C::kCols];
#pragma unroll
  for (int j = 0; j < C::kCols; ++j) sum[j] = 0.f;
  const int first = few ? 0 : item.n_kb;
  if (threadIdx.x == 0 && !few)
    for (int i = 0; i < 2 && i < item.n_kb; ++i) item.load(first + i);
  for (int i = 0; i < item.n_kb; ++i) {
    const int u = first + i;
    if (!__syncthreads_and(item.arrived(u, 6u))) {
      if (i + 1 < item.n_kb) item.arrived(u + 1, 7u);   // (under way too)
      break;
    }
    const float* const at = reinterpret_cast<const float*>(item.raw + (u & 1) * C::kRaw);
    if (mine) {
#pragma unroll 1
      for (int k = 0; k < (few ? 8 : kBK); k += 4) {   // (beyond K a block is zero)
        float c[4][4];   // [k][column]
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 v = *reinterpret_cast<const float4*>(at + c_at + (wt ? q * kBK + k : (k + q) * BN));
          if (wt)
            c[0][q] = v.x, c[1][q] = v.y, c[2][q] = v.z, c[3][q] = v.w;
          else
            c[q][0] = v.x, c[q][1] = v.y, c[q][2] = v.z, c[q][3] = v.w;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int h = 0; h < kRuns; ++h) {
            const float4 v = *reinterpret_cast<const float4*>(at + l_at + (k + q) * kLanes + h * 4 * kAlong);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              sum[h * 16 + j] = fmaf(v.x, c[q][j], sum[h * 16 + j]);
              sum[h * 16 + 4 + j] = fmaf(v.y, c[q][j], sum[h * 16 + 4 + j]);
              sum[h * 16 + 8 + j] = fmaf(v.z, c[q][j], sum[h * 16 + 8 + j]);
              sum[h * 16 + 12 + j] = fmaf(v.w, c[q][j], sum[h * 16 + 12 + j]);
            }
          }
      }
    }
    __syncthreads();
    if (threadIdx.x == 0 && i + 2 < item.n_kb) item.load(u + 2);
  }
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == kWarps) return;
  const long long l = item.l0 + (warp & 3) * 32 + run, n = item.c0 + (warp >> 2) * C::kCols + four;
#pragma unroll
  for (int h = 0; h < kRuns; ++h) {
    float v[4][4];   // [lane][column]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[i][j] = sum[h * 16 + 4 * i + j];
        if (!few) {
          const float was = old[(four + j) * kWarps * 32 + warp * 32 + h * 4 * kAlong + run + i];
          if (stays(was)) v[i][j] = was;
        }
      }
    if (l + h * 4 * kAlong >= item.lanes) continue;
#pragma unroll
    for (int i = 0; i < 4; ++i) {   // (lanes are a multiple of four, and columns where they lie together)
      if (wt && n + i < item.cols)
        *reinterpret_cast<float4*>(item.D + (n + i) * item.lanes + l + h * 4 * kAlong) = make_float4(v[0][i], v[1][i], v[2][i], v[3][i]);
      if (!wt && n < item.cols)
        *reinterpret_cast<float4*>(item.D + (l + h * 4 * kAlong + i) * item.cols + n) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
    }
  }
}

template <int BN>
__global__ void __launch_bounds__(kThreads, 1) gemm_fp32_split_kernel(const __grid_constant__ GemmFp32Jobs jobs,
                                                                    const __grid_constant__ Maps maps) {
  using C = Cfg<BN>;
  const Item<BN> item(jobs, maps);
  uint8_t *const smem = item.smem, *const raw = item.raw;
  uint64_t* const full = item.full;
  uint64_t* ready = full + 2;                                        // [2]: a block's parts are written
  uint64_t* done = ready + 2;                                        // [2]: its MMAs have completed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool wt = item.wt;
  const int n_kb = item.n_kb;
  const bool few = n_kb == 1 && item.K - static_cast<long long>(item.kb0) * kBK <= kFewTerms;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&full[i], 1);
      ptx::mbar_init(&ready[i], kWarps);
      ptx::mbar_init(&done[i], 1);
    }
    ptx::mbar_fence_init();
    ptx::prefetch_tensormap(item.map_l);
    ptx::prefetch_tensormap(item.map_c);
  }
  if (warp == 0 && !few) {
    ptx::tmem_alloc(tmem_slot, kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;   // (few: none)
  asm volatile("griddepcontrol.wait;" ::: "memory");   // launched as the kernel ahead ends

  if (few) {
    if (threadIdx.x == 0) item.load(0);
    finish_by_fma<BN>(jobs, maps, true, true);
    return;
  }
  // L: a thread has its lane's k's of one half of the block.  C: pieces of four numbers, a
  // warp whole 128-byte lines; row `row` + q * rows of the block, in shared memory `hop` apart.
  const bool is_l = warp < 8;
  const int quarter = warp & 3, tid = threadIdx.x & 255;
  const int c_row = wt ? tid >> 4 : tid / (BN / 4), c_pc = wt ? tid & 15 : tid % (BN / 4);
  const int hop = (wt ? 16 : 256 / (BN / 4)) * 128;
  const int to = (wt ? 0 : (c_pc >> 4) * kChunkBytes) + c_row * 128 + ((((c_pc & 15) >> 1) ^ (c_row & 7)) << 4) + (c_pc & 1) * 8;

  float sum[C::kCols];
#pragma unroll
  for (int j = 0; j < C::kCols; ++j) sum[j] = 0.f;
  const int group = warp >> 2;
  const uint32_t lane_bits = static_cast<uint32_t>(quarter * 32) << 16;
  const uint32_t acc_at = tmem_base + lane_bits + group * C::kCols;
  bool ok = true;
  auto drain = [&](int i) {
    ok = __all_sync(0xffffffffu,
                    ptx::mbar_wait(&done[i & 1], static_cast<uint32_t>(i >> 1) & 1u, jobs.status, (7u << 16) | 1u));
    ptx::tc_fence_after_sync();
#pragma unroll
    for (int c = 0; c < C::kCols; c += 16) {
      uint32_t a[16];
      ptx::tmem_ld_xn<16>(acc_at + (i & 1) * BN + c, a);
      ptx::tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < 16; ++j) sum[c + j] += __uint_as_float(a[j]);
    }
  };

  int begun = 0;   // blocks whose MMAs this thread has issued
  if (warp == kWarps) {
    if (ptx::elect_one()) {
      const uint32_t idesc = ptx::idesc_bf16(kLanes, BN, false, !wt);
      const int n = jobs.test_stall ? 0 : n_kb;
      int loads = 0;   // blocks fetched
      for (; loads < 2 && loads < n; ++loads) item.load(loads);
      for (int i = 0; i < n_kb; ++i) {
        const int s = i & 1;
        if (!ptx::mbar_wait(&ready[s], static_cast<uint32_t>(i >> 1) & 1u, jobs.status, (7u << 16) | 3u)) break;
        if (i + 2 < n_kb) item.load(loads++);   // everyone has read block i
        ptx::tc_fence_after_sync();
        const uint32_t a = tmem_base + kTmemL + s * 3 * kPartCols, b = ptx::smem_u32(smem + s * C::kStage);
        const uint32_t d = tmem_base + s * BN;
        // parts 0 hi, 1 mid, 2 lo.  mid * mid comes out times 2^30, the products of one of them
        // times 2^15, hi * hi as it is: the accumulator is taken down between them
        constexpr int kPl[6] = {1, 2, 0, 1, 0, 0}, kPc[6] = {1, 0, 2, 0, 1, 0};
#pragma unroll
        for (int q = 0; q < 6; ++q)
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
            const uint32_t bp = b + kPc[q] * C::kPart;
            const uint64_t db = wt ? ptx::smem_desc_sw128(bp + kk * 32, 16, 1024)
                                   : ptx::smem_desc_sw128(bp + kk * 2048, kChunkBytes, 1024);
            const uint32_t al = a + kPl[q] * kPartCols + kk * 8;
            if (kk == 0 && (q == 1 || q == 5))
              mma_bf16_ts_down(d, al, db, idesc);
            else
              mma_bf16_ts(d, al, db, idesc, (q == 0 && kk == 0) ? 0u : 1u);
          }
        ptx::mma_commit(&done[s]);
        begun = i + 1;
      }
      // (after an expired wait: no load is under way when the CTA ends)
      for (int i = begun; i < loads; ++i) item.arrived(i, 4u);
      ok = begun == n_kb;
    }
    __syncwarp();
  }
  for (int i = 0; i < n_kb && ok && warp < kWarps; ++i) {
    // (the MMAs that read this stage of parts have completed: their accumulator was drained)
    const int s = i & 1;
    ok = __all_sync(0xffffffffu, item.arrived(i, 2u));
    if (!ok) break;
    if (is_l) {
      const float* const src = reinterpret_cast<const float*>(raw + s * C::kRaw) + (warp >> 2) * 32 * kLanes + quarter * 32 + lane;
      const uint32_t dst = tmem_base + lane_bits + kTmemL + s * 3 * kPartCols + (warp >> 2) * 16;
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // 16 k's
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = src[(16 * h + j) * kLanes];
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          uint32_t w[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) w[j] = take_part(v[2 * j], v[2 * j + 1], part);
          tmem_st_x8(dst + part * kPartCols + h * 8, w);
        }
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    } else {
      const float4* const src = reinterpret_cast<const float4*>(raw + s * C::kRaw + C::kRawL) + tid;
      uint8_t* const dst = smem + s * C::kStage + to;
#pragma unroll
      for (int q = 0; q < C::kPieces; ++q) {
        float4 v = src[q * 256];
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          const uint32_t w0 = take_part(v.x, v.y, part), w1 = take_part(v.z, v.w, part);
          *reinterpret_cast<uint2*>(dst + q * hop + part * C::kPart) = make_uint2(w0, w1);
        }
      }
      ptx::fence_proxy_async_smem();   // the tensor core reads the parts through the async proxy
    }
    ptx::tc_fence_before_sync();
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(&ready[s]);
    if (i > 0) drain(i - 1);   // under the MMAs just issued
  }
  if (ok && warp < kWarps) drain(n_kb - 1);

  const long long lanes = item.lanes, cols = item.cols;
  const long long l = item.l0 + quarter * 32 + lane, n0 = item.c0 + group * C::kCols;   // this thread's lane, its columns
  float most = 0.f;
  uint32_t least = ~0u;
#pragma unroll
  for (int j = 0; j < C::kCols; j += 2) {
    // (a NaN stays; zero becomes the largest)
    asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(most) : "f"(sum[j]), "f"(sum[j + 1]));
    least = __vimin3_u32(least, __float_as_uint(sum[j]) * 2u - 1u, __float_as_uint(sum[j + 1]) * 2u - 1u);
  }
  const bool bad = !(most <= kMostSum) || least < __float_as_uint(kLeastSum) * 2u - 1u;
  ptx::tc_fence_before_sync();
  // past this barrier every load, MMA and read of TMEM and shared memory has ended, unless a wait ran out
  if (__syncthreads_or(bad || !ok)) {
    if (__syncthreads_and(ok)) {
      if (warp == 0) ptx::tmem_dealloc(tmem_base, kTmemCols);
      if (warp < kWarps) {
#pragma unroll
        for (int j = 0; j < C::kCols; ++j) reinterpret_cast<float*>(smem)[j * kWarps * 32 + threadIdx.x] = sum[j];
      }
      finish_by_fma<BN>(jobs, maps, false, __any_sync(0xffffffffu, bad));
      return;
    }
    if (begun > 0)
      ptx::mbar_wait(&done[(begun - 1) & 1], static_cast<uint32_t>((begun - 1) >> 1) & 1u, jobs.status, (7u << 16) | 5u);
    __syncthreads();
  }
  if (warp == 0) ptx::tmem_dealloc(tmem_base, kTmemCols);
  // The next kernel may start, as late as this: CTAs that come early, while some SMs are
  // idle, would all settle on those.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == kWarps) return;
  float* const D = item.D;
  if (wt) {   // a warp 32 numbers of a row at a time
#pragma unroll
    for (int j = 0; j < C::kCols; ++j)
      if (l < lanes && n0 + j < cols) D[(n0 + j) * lanes + l] = sum[j];
  } else {    // through shared memory, a warp its own 32 rows, so that a store covers whole rows
    constexpr int kRowPieces = C::kCols / 4;
    float4* const mine = reinterpret_cast<float4*>(smem) + warp * 32 * kRowPieces;
#pragma unroll
    for (int c = 0; c < kRowPieces; ++c)
      mine[lane * kRowPieces + (c ^ (lane & (kRowPieces - 1)))] =
          make_float4(sum[4 * c], sum[4 * c + 1], sum[4 * c + 2], sum[4 * c + 3]);
    __syncwarp();
    const int c = lane % kRowPieces;
#pragma unroll
    for (int r0 = 0; r0 < 32; r0 += 32 / kRowPieces) {
      const int row = r0 + lane / kRowPieces;
      const long long gm = item.l0 + quarter * 32 + row, gn = n0 + 4 * c;
      if (gm < lanes && gn < cols)
        *reinterpret_cast<float4*>(D + gm * cols + gn) = mine[row * kRowPieces + (c ^ (row & (kRowPieces - 1)))];
    }
  }
}

}  // namespace split

static thread_local bool g_test_stall = false;
void set_test_stall_fp32(bool on) { g_test_stall = on; }

template <int BN>
static int launch_bn(const GemmFp32Jobs& js, int n, cudaStream_t stream) {
  using C = split::Cfg<BN>;
  split::Maps maps;
  for (int i = 0; i < n; ++i) {
    const GemmFp32Job& g = js.j[i];
    if (g.a_mn) {
      if (int e = encode_f32_matrix_map(&maps.l[i], g.A, g.K, g.M, split::kBK, split::kLanes)) return e;
      if (int e = encode_f32_matrix_map(&maps.c[i], g.B, g.K, g.N, split::kBK, BN)) return e;
    } else {
      if (int e = encode_f32_matrix_map(&maps.l[i], g.B, g.K, g.N, split::kBK, split::kLanes)) return e;
      if (int e = encode_f32_matrix_map(&maps.c[i], g.A, g.M, g.K, BN, split::kBK)) return e;
    }
  }
  static PerDevice configured;
  const auto kern = split::gemm_fp32_split_kernel<BN>;
  if (int e = allow_dynamic_smem(configured, reinterpret_cast<const void*>(kern), C::kSmem)) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(js.items);
  cfg.blockDim = dim3(split::kThreads);
  cfg.dynamicSmemBytes = C::kSmem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  LBP_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, js, maps));
  count_launch();
  return LBP_OK;
}

int launch_gemm_fp32_split(GemmFp32Jobs& js, int n, int bn, cudaStream_t stream) {
  js.test_stall = g_test_stall ? 1 : 0;
  return bn == 64 ? launch_bn<64>(js, n, stream) : launch_bn<128>(js, n, stream);
}

}  // namespace lbp
