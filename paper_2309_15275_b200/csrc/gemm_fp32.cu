// fp32 products (Algorithm 1's two in the low-rank space, Eq. 2's two) on the FFMA pipe.
//
// fp32 data must meet a 1e-5 relative error, which a single-pass TF32 tensor
// product (10-bit mantissa) cannot.
//   D[M, N] = sum_k A(m, k) * B(k, n),  B stored (K, N) row-major,
//   A stored (M, K) row-major or, when A_MN, (K, M) row-major.
//
// Both products of a call go out in one launch: they are independent, and either alone
// leaves SMs idle.  An item of work is a 64 x 64 tile over at most `per` k-blocks of 32; a
// CTA takes one item, and where K needs several, each writes its sums to a plane of its
// own, which one more kernel adds up in order.  So the items of a small M x N with a long
// K and of a large one with a short K last equally long, and fill the chip together
// (plan(): slices through planes are taken only where they pay for themselves).
// A thread holds 8 x 4 sums; operands come by cp.async into three stages of 32 k's (A as
// it lies: from (M, K) a thread reads four k's of a row at once, from (K, M) four rows).
// What bounds it: shared-memory reads (a k-block of a tile takes an SM about 1 us, FFMA
// alone 0.54).  8 x 8 sums in 64 threads read less but leave the latency bare: 3.1 us for a
// CTA alone.  64 blocks of 448 -> 1792 at rank 10 with both products (7840 k-blocks of
// tiles) 64 -> 58 us, 48 rows of 2880 -> 960 at order 16 (2700) 140 -> 25.
#include "lbp_internal.h"
#include "ptx_sm100.cuh"

namespace lbp {

namespace {

constexpr int kTile = 64, kBK = 32, kThreads = 128, kStages = 3;
constexpr int kAStride = kBK + 4;     // (M, K) layout: floats per row
constexpr int kStageFloats = kTile * kAStride + kBK * kTile;   // A in either layout, then B
constexpr int kSmemBytes = kStages * kStageFloats * 4;
constexpr int kResident = 4;          // CTAs of an SM at a time
constexpr int kSms = 148;             // of a B200 (the scratch is sized without a device)

struct Job {
  const float *A, *B;
  float* D;                       // chunks > 1: the planes [chunks][M][N]
  long long M, N, K;
  int32_t a_mn, tiles_n, tiles;   // tiles of D along N, in all
  int32_t kb, chunks;             // k-blocks; items per tile
};
struct Jobs {
  Job j[2];
  int32_t n, per, items0;         // k-blocks of an item; items of the first job
};

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool valid) {
  const int bytes = valid ? 16 : 0;   // 0: the 16 bytes are filled with zeros, nothing is read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(smem)), "l"(gmem), "r"(bytes)
               : "memory");
}

// Row of the tile that sum i of a thread belongs to: two runs of four, 32 apart, so that
// the rows a warp reads from either layout lie in different banks.
__device__ __forceinline__ int row_of(int ty, int i) { return (i >> 2) * 32 + ty * 4 + (i & 3); }

template <bool A_MN>
__device__ __forceinline__ void tile_sums(const Job& g, long long m0, long long n0, int kb0, int kb1,
                                          float* smem, float (&acc)[8][4]) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  // what this thread fetches of a k-block: four 16-byte pieces of A and of B, each a fixed
  // stride after the one before
  const int am = A_MN ? (tid & 15) * 4 : tid >> 3, ak = A_MN ? tid >> 4 : (tid & 7) * 4;
  const int bn = (tid & 15) * 4, bk = tid >> 4;
  const long long k00 = static_cast<long long>(kb0) * kBK;
  const float* a_at = A_MN ? g.A + (k00 + ak) * g.M + m0 + am : g.A + (m0 + am) * g.K + k00 + ak;
  const float* b_at = g.B + (k00 + bk) * g.N + n0 + bn;
  const long long a_step = A_MN ? 8 * g.M : 16 * g.K, b_step = 8 * g.N;
  const bool b_in = n0 + bn < g.N, a_in = m0 + am < g.M;   // M (K, M), K (M, K) and N are multiples of 4
  const int left_m = A_MN ? 0 : static_cast<int>(g.M - m0 < kTile ? g.M - m0 : kTile);
  auto fetch = [&](int kb, int stage) {
    float* as = smem + stage * kStageFloats;
    float* bs = as + kTile * kAStride;
    const long long rest = g.K - static_cast<long long>(kb) * kBK;
    const int left_k = rest < kBK ? static_cast<int>(rest) : kBK;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      bool ok;
      if constexpr (A_MN) {   // 32 rows of 64 m
        ok = a_in && ak + 8 * i < left_k;
        cp_async16(as + (ak + 8 * i) * kTile + am, ok ? a_at + i * a_step : g.A, ok);
      } else {                // 64 rows of 32 k
        ok = am + 16 * i < left_m && ak < left_k;
        cp_async16(as + (am + 16 * i) * kAStride + ak, ok ? a_at + i * a_step : g.A, ok);
      }
      ok = b_in && bk + 8 * i < left_k;
      cp_async16(bs + (bk + 8 * i) * kTile + bn, ok ? b_at + i * b_step : g.B, ok);
    }
    a_at += A_MN ? kBK * g.M : kBK;
    b_at += kBK * g.N;
  };
  auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) {
    if (kb0 + s < kb1) fetch(kb0 + s, s);
    commit();
  }
  int stage = 0;
  for (int kb = kb0; kb < kb1; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();   // the stage has arrived for all, and all are done with the one before
    const float* as = smem + stage * kStageFloats;
    const float* bs = as + kTile * kAStride;
    if (kb + kStages - 1 < kb1) fetch(kb + kStages - 1, stage == 0 ? kStages - 1 : stage - 1);
    commit();
    stage = stage + 1 == kStages ? 0 : stage + 1;
#pragma unroll
    for (int k4 = 0; k4 < kBK; k4 += 4) {
      float a[8][4];   // [row][k]
      if constexpr (A_MN) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 lo = *reinterpret_cast<const float4*>(as + (k4 + k) * kTile + ty * 4);
          const float4 hi = *reinterpret_cast<const float4*>(as + (k4 + k) * kTile + 32 + ty * 4);
          a[0][k] = lo.x, a[1][k] = lo.y, a[2][k] = lo.z, a[3][k] = lo.w;
          a[4][k] = hi.x, a[5][k] = hi.y, a[6][k] = hi.z, a[7][k] = hi.w;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 v = *reinterpret_cast<const float4*>(as + row_of(ty, i) * kAStride + k4);
          a[i][0] = v.x, a[i][1] = v.y, a[i][2] = v.z, a[i][3] = v.w;
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 b = *reinterpret_cast<const float4*>(bs + (k4 + k) * kTile + tx * 4);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          acc[i][0] = fmaf(a[i][k], b.x, acc[i][0]);
          acc[i][1] = fmaf(a[i][k], b.y, acc[i][1]);
          acc[i][2] = fmaf(a[i][k], b.z, acc[i][2]);
          acc[i][3] = fmaf(a[i][k], b.w, acc[i][3]);
        }
      }
    }
  }
}

__global__ void __launch_bounds__(kThreads, kResident) gemm_fp32_kernel(const __grid_constant__ Jobs jobs) {
  extern __shared__ __align__(16) float smem[];
  asm volatile("griddepcontrol.wait;" ::: "memory");   // launched as the kernel ahead ends
  int t = blockIdx.x;
  const Job& g = jobs.j[t >= jobs.items0 ? 1 : 0];
  if (t >= jobs.items0) t -= jobs.items0;
  const int chunk = t % g.chunks;
  t /= g.chunks;
  const long long m0 = static_cast<long long>(t / g.tiles_n) * kTile, n0 = static_cast<long long>(t % g.tiles_n) * kTile;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  const int kb0 = chunk * jobs.per, kb1 = kb0 + jobs.per < g.kb ? kb0 + jobs.per : g.kb;
  if (g.a_mn)
    tile_sums<true>(g, m0, n0, kb0, kb1, smem, acc);
  else
    tile_sums<false>(g, m0, n0, kb0, kb1, smem, acc);
  // The next kernel may start, as late as this: CTAs that come early, while some SMs are
  // idle, would all settle on those.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  float* const D = g.D + chunk * g.M * g.N;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const long long m = m0 + row_of(ty, i), n = n0 + tx * 4;
    if (m < g.M && n < g.N)
      *reinterpret_cast<float4*>(D + m * g.N + n) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  }
}

long long tiles_of(const GemmFp32& g) {
  return ((g.M + kTile - 1) / kTile) * ((g.N + kTile - 1) / kTile);
}
long long kblocks(const GemmFp32& g) { return (g.K + kBK - 1) / kBK; }

// k-blocks of an item, and the bytes of planes that takes (at most `room`).  An SM works
// off a k-block in about a microsecond however many CTAs it holds (its shared-memory reads
// bind: 12 of 16 bytes per 32 FFMA), so what counts is how many k-blocks the fullest SM
// gets, and short items share out best: 2 to 5 k-blocks, or K left whole.  (Longer ones only
// with many items per SM: with two or three, 6 to 12 k-blocks measured up to half as slow
// again as 3 or 4.)  Planes cost their bytes and about 1.5 us of the kernel that adds them
// up.  28 tiles of 42 k-blocks and 147 of 8 (256 tokens, exact, 448 -> 1344): 53 us whole,
// 23 at 4, 34 at 8; 212 of 8 and 16 of 105: 133 whole, 50 at 4; 15 of 90 and 675 of 2: 121
// and 42; 12 of 12 and 12 of 11: 14 whole, 16 at 4.
long long plan(const GemmFp32* job, int n, size_t room, size_t* planes) {
  constexpr size_t kRoom = 48u << 20;
  if (room > kRoom) room = kRoom;
  long long most = 1;
  for (int i = 0; i < n; ++i) most = kblocks(job[i]) > most ? kblocks(job[i]) : most;
  long long best = most;
  double best_t = -1.0;
  *planes = 0;
  for (long long per : {most, 64ll, 32ll, 16ll, 8ll, 5ll, 4ll, 3ll, 2ll}) {
    if (per > most) continue;
    double items = 0, t = 0;
    size_t bytes = 0;
    for (int i = 0; i < n; ++i) {
      const long long chunks = (kblocks(job[i]) + per - 1) / per;
      items += static_cast<double>(tiles_of(job[i])) * chunks;
      if (chunks > 1) {
        const size_t b = static_cast<size_t>(chunks) * job[i].M * job[i].N * 4;
        bytes += b;
        t += 1.5 + 2.0 * b / 8e6;
      }
    }
    if (bytes > room || (per > 5 && per < most && items < 8.0 * kSms)) continue;
    t += static_cast<double>(static_cast<long long>((items + kSms - 1) / kSms)) * (per + 0.2);
    if (best_t < 0 || t < best_t) {
      best_t = t;
      best = per;
      *planes = bytes;
    }
  }
  return best;
}

}  // namespace

size_t gemm_fp32_ws_bytes(const GemmFp32* job, int n) {
  size_t planes = 0;
  plan(job, n, static_cast<size_t>(-1), &planes);
  return planes;
}

int launch_gemm_fp32(const GemmFp32* job, int n, float* ws, size_t ws_bytes, cudaStream_t stream) {
  Jobs js{};
  js.n = n;
  size_t planes = 0;
  const long long per = plan(job, n, ws != nullptr ? ws_bytes : 0, &planes);
  long long items = 0;
  for (int i = 0; i < n; ++i) {
    const long long tiles = tiles_of(job[i]), kb = kblocks(job[i]), chunks = (kb + per - 1) / per;
    if (tiles >= (1ll << 30) || kb >= (1ll << 30) || items + tiles * chunks >= (1ll << 31)) return LBP_ERR_SHAPE;
    js.j[i] = Job{job[i].A, job[i].B, chunks > 1 ? ws : job[i].D, job[i].M, job[i].N, job[i].K, job[i].a_mn ? 1 : 0,
                  static_cast<int32_t>((job[i].N + kTile - 1) / kTile), static_cast<int32_t>(tiles),
                  static_cast<int32_t>(kb), static_cast<int32_t>(chunks)};
    if (chunks > 1) ws += chunks * job[i].M * job[i].N;
    items += tiles * chunks;
    if (i == 0) js.items0 = static_cast<int32_t>(items);
  }
  js.per = static_cast<int32_t>(per);
  static PerDevice configured;
  if (int e = allow_dynamic_smem(configured, reinterpret_cast<const void*>(gemm_fp32_kernel), kSmemBytes)) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(items));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  LBP_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_fp32_kernel, js));
  count_launch();
  for (int i = 0; i < n; ++i)
    if (js.j[i].chunks > 1)
      if (int e = launch_splitk_reduce(js.j[i].D, job[i].D, job[i].M * job[i].N, js.j[i].chunks, false, 0.f, true, stream))
        return e;
  return LBP_OK;
}

}  // namespace lbp
