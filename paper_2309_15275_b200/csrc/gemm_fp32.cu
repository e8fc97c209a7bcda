// fp32 products (Algorithm 1's two in the low-rank space, Eq. 2's two): the plan, and the
// kernel on the FFMA pipe for the smallest of them (the others: gemm_fp32_split.cu).
//
//   D[M, N] = sum_k A(m, k) * B(k, n),  B stored (K, N) row-major,
//   A stored (M, K) row-major or, when A_MN, (K, M) row-major.
//
// Both products of a call go out in one launch: they are independent, and either alone
// leaves SMs idle.  An item of work is a tile over a run of k-blocks; a CTA takes one item,
// and where K needs several, each writes its sums to a plane of its own, which one more
// kernel adds up in order.  So the items of a small M x N with a long K and of a large one
// with a short K last equally long, and fill the chip together (plan(): slices through planes
// are taken only where they pay for themselves).
//
// FFMA kernel: tiles of 64 x 64, k-blocks of 32.  A thread holds 8 x 4 sums; operands come by
// cp.async into three stages (A as it lies: from (M, K) a thread reads four k's of a row at
// once, from (K, M) four rows).  What bounds it: shared-memory reads (a k-block of a tile takes
// an SM about 1 us, FFMA alone 0.54).  8 x 8 sums in 64 threads read less but leave the latency
// bare: 3.1 us for a CTA alone.
#include <cstdio>

#include "gemm_fp32.cuh"
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

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool valid) {
  const int bytes = valid ? 16 : 0;   // 0: the 16 bytes are filled with zeros, nothing is read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_u32(smem)), "l"(gmem), "r"(bytes)
               : "memory");
}

// Row of the tile that sum i of a thread belongs to: two runs of four, 32 apart, so that
// the rows a warp reads from either layout lie in different banks.
__device__ __forceinline__ int row_of(int ty, int i) { return (i >> 2) * 32 + ty * 4 + (i & 3); }

template <bool A_MN>
__device__ __forceinline__ void tile_sums(const GemmFp32Job& g, long long m0, long long n0, int kb0, int kb1,
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

__global__ void __launch_bounds__(kThreads, kResident) gemm_fp32_kernel(const __grid_constant__ GemmFp32Jobs jobs) {
  extern __shared__ __align__(16) float smem[];
  asm volatile("griddepcontrol.wait;" ::: "memory");   // launched as the kernel ahead ends
  int t = blockIdx.x;
  const GemmFp32Job& g = jobs.j[t >= jobs.items0 ? 1 : 0];
  if (t >= jobs.items0) t -= jobs.items0;
  const int chunk = t % g.chunks;
  t /= g.chunks;
  const long long m0 = static_cast<long long>(t / g.tiles_c) * kTile, n0 = static_cast<long long>(t % g.tiles_c) * kTile;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  const int kb0 = chunk * g.per, kb1 = kb0 + g.per < g.kb ? kb0 + g.per : g.kb;
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

// The forms a product can take: tile, k-block, and what a k-block and an item take an SM (us).
// FFMA: an SM works off a k-block in about a microsecond however many CTAs it holds.  Split
// operands (one CTA to an SM): fitted to whole calls, in which all SMs fetch at once; alone on
// the chip a block takes 1.04 and 1.3 us, an item's start and end with the launch 5.6 and 7.
// Both sides of the line (us a call, replayed from a graph; FFMA / split, its better tile): 2 x
// 16 x 16 tokens of 64 -> 64, order 8, rank 4: 8.8 / 10.1; 8 x 7 x 7 of 64 -> 256, order 4, rank 6:
// 11.5 / 13.1; 2 x 56 x 56 of 64 -> 64, order 4, rank 6: 11.2 / 12.2; 8 x 28 x 28 of 96 -> 384, order
// 4, rank 3: 20.6 / 16.8; 8 x 56 x 56 of 48 -> 192, order 4, rank 3: 24.2 / 19.9; 8 x 28 x 28 of 192
// -> 768, order 8, rank 21: 65 / 36; 64 x 7 x 7 of 448 -> 1792, order 8, rank 10: 69 / 32; 392 tokens
// of 448 -> 1792, exact: 45 / 18.  Close to the line, where planes decide, the model is off by up
// to 2 us: it takes FFMA for 4 x 56 x 56 of 48 -> 192, rank 3 (18.0 / 16.4) and 16 x 28 x 28 of 96
// -> 96, rank 3 (15.7 / 14.1).
struct Form {
  int lanes, cols, bk;   // (split operands: lanes of TMEM, of the operand stored (K, lanes))
  double kb_us, item_us, launch_us;
};
constexpr Form kForms[] = {
    {kTile, kTile, kBK, 1.0, 0.2, 0.0},
    {128, 64, 64, 1.05, 2.5, 2.0},
    {128, 128, 64, 1.45, 3.5, 2.0},
};

struct Plan {
  int form;
  long long per;
  size_t planes;   // bytes
};

long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }
long long lanes_of(const GemmFp32& g, const Form& f) { return ceil_div(g.a_mn ? g.M : g.N, f.lanes); }
long long cols_of(const GemmFp32& g, const Form& f) { return ceil_div(g.a_mn ? g.N : g.M, f.cols); }
long long tiles_of(const GemmFp32& g, const Form& f) { return lanes_of(g, f) * cols_of(g, f); }

// Time until the last of n0 items of t0 and then n1 of t1 ends, each taken by the first SM that is free.
double makespan(long long n0, double t0, long long n1, double t1) {
  const long long q = n0 / kSms, more = n0 % kSms;
  double low = q * t0, high = low + (more > 0 ? t0 : 0.0);   // `more` SMs are free at `high`, the others at `low`
  double end = high;
  long long at_low = kSms - more, at_high = more;
  while (n1 > 0) {
    if (at_high > 0 && high < low) {
      const double d = high;
      high = low, low = d;
      const long long n = at_high;
      at_high = at_low, at_low = n;
    }
    n1 -= at_low;
    low += t1;
    end = low > end ? low : end;
  }
  return end;
}

// Items of a product of kb k-blocks at `per` an item, evenly long.
long long chunks_of(long long kb, long long per) { return ceil_div(kb, ceil_div(kb, ceil_div(kb, per))); }

// The form, k-blocks of an item, and the bytes of planes that takes (at most `room`).  FFMA:
// what counts is how many k-blocks the fullest SM gets, and short items share out best: 2 to 5
// k-blocks, or K left whole.  (Longer ones only with many items per SM: with two or three, 6
// to 12 k-blocks measured up to half as slow again as 3 or 4.)  Planes cost their bytes and
// about 1.5 us of the kernel that adds them up.
Plan make_plan(const GemmFp32* job, int n, size_t room) {
  constexpr size_t kRoom = 48u << 20;
  if (room > kRoom) room = kRoom;
  Plan best{};
  double best_t = -1.0;
  bool fits = true;   // TMA coordinates are 32-bit
  for (int i = 0; i < n; ++i)
    for (long long d : {job[i].M, job[i].N, job[i].K}) fits &= d < (1ll << 31) - 256;
  const int forced = fits ? tune_options().fp32_form : 0;
  const long long wanted = tune_options().fp32_per;
  for (int f = 0; f < 3; ++f) {
    const Form& form = kForms[f];
    if (forced >= 0 && f != forced) continue;
    long long kb[2] = {0, 0}, most = 1;
    for (int i = 0; i < n; ++i) {
      kb[i] = ceil_div(job[i].K, form.bk);
      most = kb[i] > most ? kb[i] : most;
    }
    for (long long per : {most, wanted, 64ll, 48ll, 32ll, 24ll, 16ll, 12ll, 10ll, 8ll, 7ll, 6ll, 5ll, 4ll, 3ll, 2ll, 1ll}) {
      if (per == 0 || per > most || (f == 0 && per == 1 && per < most)) continue;
      double t = 0, item_t[2] = {0, 0};
      long long items[2] = {0, 0};
      size_t bytes = 0;
      for (int i = 0; i < n; ++i) {
        const long long chunks = chunks_of(kb[i], per);
        items[i] = tiles_of(job[i], form) * chunks;
        item_t[i] = ceil_div(kb[i], chunks) * form.kb_us + form.item_us;
        if (chunks > 1) {
          const size_t b = static_cast<size_t>(chunks) * job[i].M * job[i].N * 4;
          bytes += b;
          t += 1.5 + 2.0 * b / 8e6;
        }
      }
      const double all = static_cast<double>(items[0] + items[1]);
      if (bytes > room || (f == 0 && per > 5 && per < most && all < 8.0 * kSms)) continue;
      t += f == 0 ? static_cast<double>(ceil_div(items[0] + items[1], kSms)) * (per + form.item_us)
           : item_t[0] < item_t[1] ? form.launch_us + makespan(items[1], item_t[1], items[0], item_t[0])
                                    : form.launch_us + makespan(items[0], item_t[0], items[1], item_t[1]);
      if (per == wanted) {   // whatever it takes
        best = Plan{f, per, bytes};
        break;
      }
      if (best_t < 0 || t < best_t) {
        best_t = t;
        best = Plan{f, per, bytes};
      }
    }
  }
  return best;
}

// (remembered per calling thread for recent shapes)
Plan plan(const GemmFp32* job, int n, size_t room) {
  struct Entry {
    long long dims[6];
    size_t room;
    int forced, wanted;
    Plan plan;
  };
  static thread_local Entry cache[16];
  static thread_local int filled = 0, next = 0;
  const GemmFp32 &a = job[0], &b = job[n - 1];
  const long long dims[6] = {a.M, a.N, a.K, n > 1 ? b.M : 0, n > 1 ? b.N : 0, n > 1 ? b.K : 0};
  for (int c = 0; c < filled; ++c) {
    const Entry& e = cache[c];
    bool same = e.room == room && e.forced == tune_options().fp32_form && e.wanted == tune_options().fp32_per;
    for (int i = 0; i < 6; ++i) same &= e.dims[i] == dims[i];
    if (same) return e.plan;
  }
  Entry& e = cache[next];
  for (int i = 0; i < 6; ++i) e.dims[i] = dims[i];
  e.room = room;
  e.forced = tune_options().fp32_form;
  e.wanted = tune_options().fp32_per;
  e.plan = make_plan(job, n, room);
  if (tune_options().verbose)
    fprintf(stderr, "lbp fp32 products plan: %lldx%lldx%lld, %lldx%lldx%lld: form %d, %lld k-blocks an item, planes %zu\n",
            dims[0], dims[1], dims[2], dims[3], dims[4], dims[5], e.plan.form, e.plan.per, e.plan.planes);
  next = (next + 1) % 16;
  filled = filled < 16 ? filled + 1 : 16;
  return e.plan;
}

}  // namespace

size_t gemm_fp32_ws_bytes(const GemmFp32* job, int n) {
  return plan(job, n, static_cast<size_t>(-1)).planes;
}

void gemm_fp32_plan(const GemmFp32 (&job)[2], size_t room, int64_t* out6) {
  const Plan pl = plan(job, 2, room);
  out6[0] = pl.form;
  out6[1] = static_cast<int64_t>(pl.planes);
  for (int i = 0; i < 2; ++i) {
    const long long kb = ceil_div(job[i].K, kForms[pl.form].bk), chunks = chunks_of(kb, pl.per);
    out6[2 + 2 * i] = ceil_div(kb, chunks);
    out6[3 + 2 * i] = chunks;
  }
}

int launch_gemm_fp32(const GemmFp32* job, int n, float* ws, size_t ws_bytes, uint32_t* status, cudaStream_t stream) {
  GemmFp32Jobs js{};
  js.status = status;
  const Plan pl = plan(job, n, ws != nullptr ? ws_bytes : 0);
  const Form& form = kForms[pl.form];
  // split operands: the longer items first
  const auto per_of = [&](int i) {
    const long long kb = ceil_div(job[i].K, form.bk);
    return ceil_div(kb, chunks_of(kb, pl.per));
  };
  const bool swap = n > 1 && pl.form > 0 && per_of(0) < per_of(1);
  long long items = 0;
  for (int at = 0; at < n; ++at) {
    const GemmFp32& g = job[swap ? 1 - at : at];
    const long long tiles = tiles_of(g, form), kb = ceil_div(g.K, form.bk), chunks = chunks_of(kb, pl.per);
    if (tiles >= (1ll << 30) || kb >= (1ll << 30) || items + tiles * chunks >= (1ll << 31)) return LBP_ERR_SHAPE;
    js.j[at] = GemmFp32Job{g.A, g.B, chunks > 1 ? ws : g.D, g.M, g.N, g.K, g.a_mn ? 1 : 0,
                           static_cast<int32_t>(pl.form > 0 ? cols_of(g, form) : ceil_div(g.N, form.cols)),
                           static_cast<int32_t>(tiles), static_cast<int32_t>(kb),
                           static_cast<int32_t>(ceil_div(kb, chunks)), static_cast<int32_t>(chunks)};
    if (chunks > 1) ws += chunks * g.M * g.N;
    items += tiles * chunks;
    if (at == 0) js.items0 = static_cast<int32_t>(items);
  }
  js.items = static_cast<int32_t>(items);
  if (pl.form > 0) {
    if (int e = launch_gemm_fp32_split(js, n, form.cols, stream)) return e;
  } else {
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
  }
  for (int at = 0; at < n; ++at) {
    const GemmFp32& g = job[swap ? 1 - at : at];
    if (js.j[at].chunks > 1)
      if (int e = launch_splitk_reduce(js.j[at].D, g.D, g.M * g.N, js.j[at].chunks, false, 0.f, true, stream)) return e;
  }
  return LBP_OK;
}

}  // namespace lbp
