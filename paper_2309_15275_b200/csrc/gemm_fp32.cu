// fp32 products (Algorithm 1's two in the low-rank space, Eq. 2's two) on the FFMA pipe.
//
// fp32 data must meet a 1e-5 relative error, which a single-pass TF32 tensor
// product (10-bit mantissa) cannot.
//   D[M, N] = sum_k A(m, k) * B(k, n),  B stored (K, N) row-major,
//   A stored (M, K) row-major or, when A_MN, (K, M) row-major.
//
// Both products of a call go out in one launch: they are independent, and either alone
// leaves SMs idle.  A CTA computes a 64 x 64 tile over one slice of K; the slices of a
// tile are the CTAs of a cluster (up to 8), which add their sums up through distributed
// shared memory, each CTA its share of the rows, in the order of the slices.  So a small
// M x N with a long K fills the chip without scratch and with a fixed order of sums.
// A thread holds 8 x 4 sums; operands come by cp.async into two stages of 32 k's (A as it
// lies: from (M, K) a thread reads four k's of a row at once, from (K, M) four rows).
// What bounds it: FFMA issue (128 a cycle and SM).  1792 x 448 x 640 and 640 x 448 x 1792
// (2.06 GFLOP, 28 us at the FFMA peak): 55 + 124 us in two launches of one CTA per tile
// and scalar loads.
#include "lbp_internal.h"
#include "ptx_sm100.cuh"

namespace lbp {

namespace {

constexpr int kTile = 64, kBK = 32, kThreads = 128;
constexpr int kAStride = kBK + 4;     // (M, K) layout: floats per row
constexpr int kStageFloats = kTile * kAStride + kBK * kTile;   // A in either layout, then B

struct Job {
  const float *A, *B;
  float* D;
  long long M, N, K;
  int32_t a_mn, tiles_n, tiles;   // tiles of D along N, in all
  int32_t kb, kb_per;             // k-blocks, and per slice
};
struct Jobs {
  Job j[2];
  int32_t n;
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
  auto fetch = [&](int kb, int stage) {
    float* as = smem + stage * kStageFloats;
    float* bs = as + kTile * kAStride;
    const long long k0 = static_cast<long long>(kb) * kBK;
#pragma unroll
    for (int i = 0; i < kTile * kBK / 4 / kThreads; ++i) {
      const int e = tid + i * kThreads;
      if constexpr (A_MN) {   // 32 rows of 64 m
        const int kk = e >> 4, mm = (e & 15) * 4;
        const bool ok = k0 + kk < g.K && m0 + mm < g.M;   // M is a multiple of 4
        cp_async16(as + kk * kTile + mm, ok ? g.A + (k0 + kk) * g.M + m0 + mm : g.A, ok);
      } else {                // 64 rows of 32 k
        const int mm = e >> 3, kk = (e & 7) * 4;
        const bool ok = m0 + mm < g.M && k0 + kk < g.K;   // K is a multiple of 4
        cp_async16(as + mm * kAStride + kk, ok ? g.A + (m0 + mm) * g.K + k0 + kk : g.A, ok);
      }
      const int kk = e >> 4, nn = (e & 15) * 4;
      const bool ok = k0 + kk < g.K && n0 + nn < g.N;     // N is a multiple of 4
      cp_async16(bs + kk * kTile + nn, ok ? g.B + (k0 + kk) * g.N + n0 + nn : g.B, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (kb0 < kb1) fetch(kb0, 0);
  for (int kb = kb0; kb < kb1; ++kb) {
    const int stage = (kb - kb0) & 1;
    if (kb + 1 < kb1) {
      fetch(kb + 1, stage ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float* as = smem + stage * kStageFloats;
    const float* bs = as + kTile * kAStride;
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
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kThreads) gemm_fp32_kernel(const __grid_constant__ Jobs jobs) {
  __shared__ __align__(16) float smem[2 * kStageFloats];
  const int slices = gridDim.y, slice = blockIdx.y;   // the cluster lies along y
  int t = blockIdx.x;
  const Job& g = jobs.j[t >= jobs.j[0].tiles ? 1 : 0];
  if (t >= jobs.j[0].tiles) t -= jobs.j[0].tiles;
  const long long m0 = static_cast<long long>(t / g.tiles_n) * kTile, n0 = static_cast<long long>(t % g.tiles_n) * kTile;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  const int kb0 = slice * g.kb_per, kb1 = kb0 + g.kb_per < g.kb ? kb0 + g.kb_per : g.kb;
  if (g.a_mn)
    tile_sums<true>(g, m0, n0, kb0, kb1, smem, acc);
  else
    tile_sums<false>(g, m0, n0, kb0, kb1, smem, acc);

  auto store = [&](int row, float4 v) {
    const long long m = m0 + row, n = n0 + tx * 4;
    if (m < g.M && n < g.N) *reinterpret_cast<float4*>(g.D + m * g.N + n) = v;
  };
  if (slices == 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i) store(row_of(ty, i), make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
    return;
  }
  // the tile of this slice to shared memory (the operand stages are done with)
#pragma unroll
  for (int i = 0; i < 8; ++i)
    *reinterpret_cast<float4*>(smem + row_of(ty, i) * kTile + tx * 4) =
        make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  const int rows = kTile / slices;   // this CTA adds up rows slice * rows ..
  for (int r = ty; r < rows; r += 8) {
    const int row = slice * rows + r;
    const uint32_t at = ptx::smem_u32(smem + row * kTile + tx * 4);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c = 0; c < slices; ++c) {
      float4 v;
      asm volatile(
          "{\n\t.reg .b32 p;\n\tmapa.shared::cluster.u32 p, %4, %5;\n\t"
          "ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [p];\n\t}"
          : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
          : "r"(at), "r"(c)
          : "memory");
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    }
    store(row, s);
  }
  // no CTA leaves while its sums may still be read
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace

int launch_gemm_fp32(const GemmFp32* job, int n, cudaStream_t stream) {
  Jobs js{};
  js.n = n;
  long long tiles = 0;
  int kb_most = 1;
  for (int i = 0; i < n; ++i) {
    Job& g = js.j[i];
    const long long tm = (job[i].M + kTile - 1) / kTile, tn = (job[i].N + kTile - 1) / kTile;
    const long long kb = (job[i].K + kBK - 1) / kBK;
    if (tm * tn >= (1ll << 30) || kb >= (1ll << 30)) return LBP_ERR_SHAPE;
    g = Job{job[i].A, job[i].B, job[i].D, job[i].M, job[i].N, job[i].K, job[i].a_mn ? 1 : 0,
            static_cast<int32_t>(tn), static_cast<int32_t>(tm * tn), static_cast<int32_t>(kb), 0};
    tiles += g.tiles;
    if (g.kb > kb_most) kb_most = g.kb;
  }
  int dev = 0, sms = 0;
  LBP_CUDA_TRY(cudaGetDevice(&dev));
  LBP_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // slices until there are four CTAs per SM (a CTA alone on an SM issues at a third of its
  // rate), as long as the longer product keeps two k-blocks per slice
  int slices = 1;
  while (slices < 8 && tiles * slices < 4ll * sms && kb_most >= 4 * slices) slices *= 2;
  for (int i = 0; i < n; ++i) js.j[i].kb_per = (js.j[i].kb + slices - 1) / slices;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(tiles), static_cast<unsigned>(slices));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = static_cast<unsigned>(slices);
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = slices > 1 ? 1 : 0;
  LBP_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_fp32_kernel, js));
  count_launch();
  return LBP_OK;
}

}  // namespace lbp
