// Small kernels around Algorithm 1 that a ViT layer needs and the paper leaves
// out: accumulation into g_W (outside the products kernel), the bias gradient, and
// dense copies of strided token tensors.
#include <cuda_bf16.h>

#include <algorithm>

#include "lbp_internal.h"
#include "wht_device.cuh"

namespace lbp {

namespace {

// g_W <- beta * g_W + a (+ b):  a, b fp32 (Cout x Cin), g_W fp32 or bf16.
__global__ void __launch_bounds__(256)
    gw_combine_kernel(void* __restrict__ g_W, int gw_bf16, const float* __restrict__ a,
                      const float* __restrict__ b, float beta, long long n4) {
  const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  float4 v = reinterpret_cast<const float4*>(a)[i];
  if (b != nullptr) {
    const float4 w = reinterpret_cast<const float4*>(b)[i];
    v.x += w.x;
    v.y += w.y;
    v.z += w.z;
    v.w += w.w;
  }
  if (gw_bf16) {
    uint2* dst = reinterpret_cast<uint2*>(g_W) + i;
    if (beta != 0.f) {
      const uint2 old = *dst;
      v.x = fmaf(beta, __uint_as_float(old.x << 16), v.x);
      v.y = fmaf(beta, __uint_as_float(old.x & 0xffff0000u), v.y);
      v.z = fmaf(beta, __uint_as_float(old.y << 16), v.z);
      v.w = fmaf(beta, __uint_as_float(old.y & 0xffff0000u), v.w);
    }
    *dst = make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
  } else {
    float4* dst = reinterpret_cast<float4*>(g_W) + i;
    if (beta != 0.f) {
      const float4 old = *dst;
      v.x = fmaf(beta, old.x, v.x);
      v.y = fmaf(beta, old.y, v.y);
      v.z = fmaf(beta, old.z, v.z);
      v.w = fmaf(beta, old.w, v.w);
    }
    *dst = v;
  }
}

// Gradient of a bias:  g_bias <- beta * g_bias + scale * sum of n_a rows of `a` + sum
// of n_b rows of `b`, in fp64, one launch.  Row i of `a` is the DC coefficient of
// block i of a dense coefficient matrix (r > 0: matrix row i * r + q) or, r == 0, token
// i of a tensor laid out as `ta` says; row i of `b` is token i under `tb`.
// A CTA takes 128 bytes of channels, a thread 16 of them of every 32nd row; the CTAs of
// a cluster (along y) share the rows and the first adds up their sums from shared
// memory in a fixed order.  What bounds it: latency (a few hundred rows), so rows are
// fetched four at a time and the cluster grows with their number; the three launches it
// replaces (column sums of 256 rows per CTA, of the extra tokens, and a finish) took
// 11.4 + 4.7 + 2.1 us on 256 blocks of 3072 channels and 64 class tokens.  Over many rows
// (all tokens of g_y) a few CTAs would be bound by their own loads: there are several
// clusters then, each leaves its sums in a row of `partial`, and bias_finish_kernel adds
// those up in order.  What that takes beside the call without a bias, against one cluster
// and against the three launches: 200704 tokens of 192 bf16 channels 45 us (479, 260), 32768
// of 768 32 (84, 102), 802816 of 16 129 (1149, 693).
__device__ __forceinline__ void store_bias(void* g_bias, int c, double s, int out_bf16, float beta) {
  if (out_bf16) {
    __nv_bfloat16* o = static_cast<__nv_bfloat16*>(g_bias) + c;
    if (beta != 0.f) s += static_cast<double>(beta) * static_cast<double>(__bfloat162float(*o));
    *o = __float2bfloat16_rn(static_cast<float>(s));
  } else {
    float* o = static_cast<float*>(g_bias) + c;
    if (beta != 0.f) s += static_cast<double>(beta) * static_cast<double>(*o);
    *o = static_cast<float>(s);
  }
}

template <typename T>
__global__ void __launch_bounds__(256)
    bias_grad_kernel(const T* __restrict__ a, long long n_a, int r, int q, TokenMap ta, double scale,
                     const T* __restrict__ b, long long n_b, TokenMap tb, int C, int slabs,
                     double* __restrict__ partial, void* __restrict__ g_bias, int out_bf16, float beta) {
  constexpr int V = 16 / sizeof(T);          // channels per thread
  constexpr int kCols = 8 * V;
  __shared__ double sm[32][kCols + 1];
  __shared__ double part[kCols];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int col = threadIdx.x & 7, ph = threadIdx.x >> 3;
  const int c = blockIdx.x * kCols + col * V;
  double acc[V];
#pragma unroll
  for (int v = 0; v < V; ++v) acc[v] = 0.0;
  auto add = [&](uint4 w, double f) {
    if constexpr (sizeof(T) == 2) {
      const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        acc[2 * v] += f * static_cast<double>(bf16_lo(u[v]));
        acc[2 * v + 1] += f * static_cast<double>(bf16_hi(u[v]));
      }
    } else {
      acc[0] += f * static_cast<double>(__uint_as_float(w.x));
      acc[1] += f * static_cast<double>(__uint_as_float(w.y));
      acc[2] += f * static_cast<double>(__uint_as_float(w.z));
      acc[3] += f * static_cast<double>(__uint_as_float(w.w));
    }
  };
  if (c < C) {   // C is a multiple of V
    const long long first = static_cast<long long>(blockIdx.y) * 32 + ph, step = 32ll * gridDim.y;
    constexpr int U = 4;
    for (long long i = first; i < n_a; i += U * step) {
      uint4 w[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const long long j = i + u * step;
        w[u] = make_uint4(0u, 0u, 0u, 0u);
        if (j < n_a)
          w[u] = *reinterpret_cast<const uint4*>(
              a + (r > 0 ? (j * r + q) * static_cast<long long>(C) : ta.offset(j)) + c);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) add(w[u], scale);
    }
    for (long long i = first; i < n_b; i += step)
      add(*reinterpret_cast<const uint4*>(b + tb.offset(i) + c), 1.0);
  }
#pragma unroll
  for (int v = 0; v < V; ++v) sm[ph][col * V + v] = acc[v];
  __syncthreads();
  if (threadIdx.x < kCols) {
    double s = 0.0;
#pragma unroll 8
    for (int j = 0; j < 32; ++j) s += sm[j][threadIdx.x];   // fixed order
    part[threadIdx.x] = s;
  }
  if (slabs > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
  const int cc = blockIdx.x * kCols + threadIdx.x;
  uint32_t rank;   // in the cluster
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  if (rank == 0 && threadIdx.x < kCols && cc < C) {
    double s = part[threadIdx.x];
    for (int j = 1; j < slabs; ++j) {
      uint32_t at = static_cast<uint32_t>(__cvta_generic_to_shared(&part[threadIdx.x]));
      double o;
      asm volatile(
          "{\n\t.reg .b32 t;\n\tmapa.shared::cluster.u32 t, %1, %2;\n\tld.shared::cluster.f64 %0, [t];\n\t}"
          : "=d"(o)
          : "r"(at), "r"(j)
          : "memory");
      s += o;
    }
    if (partial != nullptr)
      partial[static_cast<long long>(blockIdx.y / slabs) * C + cc] = s;
    else
      store_bias(g_bias, cc, s, out_bf16, beta);
  }
  if (slabs > 1)   // no CTA leaves while its sums may still be read
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// g_bias <- beta * g_bias + the sum of `rows` rows of partial sums: 32 channels a block, eight
// threads a channel.
__global__ void __launch_bounds__(256)
    bias_finish_kernel(const double* __restrict__ partial, int rows, int C, void* __restrict__ g_bias, int out_bf16,
                       float beta) {
  __shared__ double sm[8][32];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lane = threadIdx.x & 31, ph = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (c < C)
    for (int i = ph; i < rows; i += 8) s += partial[static_cast<long long>(i) * C + c];
  sm[ph][lane] = s;
  __syncthreads();
  if (ph != 0 || c >= C) return;
  for (int j = 1; j < 8; ++j) s += sm[j][lane];
  store_bias(g_bias, c, s, out_bf16, beta);
}

// Moves n_tok tokens of C channels between a tensor laid out as `tm` says and a
// dense (n_tok, C) matrix; one thread moves 16 bytes.  Strides in 16-byte units.
__global__ void __launch_bounds__(256)
    copy_tokens_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, long long n_vec,
                       int row_vec, TokenMap tm16, int to_dense) {
  const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n_vec) return;
  const long long tok = i / row_vec;
  const int piece = static_cast<int>(i - tok * row_vec);
  const long long far = tm16.offset(tok) + piece;
  if (to_dense)
    dst[i] = src[far];
  else
    dst[far] = src[i];
}

}  // namespace

int launch_copy_tokens(const void* src, void* dst, bool to_dense, long long n_tok, int C, int dtype,
                       TokenMap tm, cudaStream_t stream) {
  if (n_tok <= 0) return LBP_OK;
  const int es = dtype == LBP_BF16 ? 2 : 4;
  const int per = 16 / es;   // elements per 16 bytes; every stride is a multiple of it
  const int row_vec = C / per;
  TokenMap tm16{tm.HW, tm.W, tm.s_image / per, tm.s_row / per, tm.s_tok / per};
  const long long n_vec = n_tok * row_vec;
  copy_tokens_kernel<<<static_cast<unsigned>((n_vec + 255) / 256), 256, 0, stream>>>(
      static_cast<const uint4*>(src), static_cast<uint4*>(dst), n_vec, row_vec, tm16, to_dense ? 1 : 0);
  count_launch();
  LBP_CUDA_TRY(cudaGetLastError());
  return LBP_OK;
}

int launch_gw_combine(void* g_W, bool gw_bf16, const float* a, const float* b, float beta,
                      long long mn, cudaStream_t stream) {
  const long long n4 = mn / 4;   // Cin * element size is a multiple of 16 bytes, so mn % 4 == 0
  gw_combine_kernel<<<static_cast<unsigned>((n4 + 255) / 256), 256, 0, stream>>>(
      g_W, gw_bf16 ? 1 : 0, a, b, beta, n4);
  count_launch();
  LBP_CUDA_TRY(cudaGetLastError());
  return LBP_OK;
}

int launch_bias_grad(const void* a, long long n_a, int r, int q, TokenMap ta, double scale,
                     const void* b, long long n_b, TokenMap tb, int C, int dtype, void* g_bias,
                     bool out_bf16, float beta, double* scratch, size_t scratch_bytes, cudaStream_t stream) {
  const int cols = dtype == LBP_BF16 ? 64 : 32, tiles = (C + cols - 1) / cols;
  // a slab of at least 128 rows: four fetches per thread
  int slabs = 1;
  while (slabs < 8 && 128ll * slabs < n_a + n_b) slabs *= 2;
  // Clusters that share the rows: up to four CTAs an SM in all, 2048 rows a cluster at the least
  // (with fewer the second launch costs more than it gives).
  long long clusters = 1;
  if (slabs == 8 && n_a + n_b >= 4096) {
    const long long fit = static_cast<long long>(scratch_bytes / (static_cast<size_t>(C) * 8));
    clusters = std::min({(n_a + n_b) / 2048, (4ll * 148 + 8 * tiles - 1) / (8 * tiles), fit});
    if (clusters < 2) clusters = 1;
  }
  double* const partial = clusters > 1 ? scratch : nullptr;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(tiles), static_cast<unsigned>(slabs * clusters));
  cfg.blockDim = dim3(256);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = static_cast<unsigned>(slabs);
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = slabs > 1 ? 2 : 1;
  if (dtype == LBP_BF16)
    LBP_CUDA_TRY(cudaLaunchKernelEx(&cfg, bias_grad_kernel<__nv_bfloat16>, static_cast<const __nv_bfloat16*>(a),
                                    n_a, r, q, ta, scale, static_cast<const __nv_bfloat16*>(b), n_b, tb, C,
                                    slabs, partial, g_bias, out_bf16 ? 1 : 0, beta));
  else
    LBP_CUDA_TRY(cudaLaunchKernelEx(&cfg, bias_grad_kernel<float>, static_cast<const float*>(a), n_a, r, q, ta,
                                    scale, static_cast<const float*>(b), n_b, tb, C, slabs, partial, g_bias,
                                    out_bf16 ? 1 : 0, beta));
  count_launch();
  if (partial != nullptr) {
    cfg.gridDim = dim3(static_cast<unsigned>((C + 31) / 32));
    cfg.numAttrs = 1;
    LBP_CUDA_TRY(cudaLaunchKernelEx(&cfg, bias_finish_kernel, static_cast<const double*>(partial),
                                    static_cast<int>(clusters), C, g_bias, out_bf16 ? 1 : 0, beta));
    count_launch();
  }
  return LBP_OK;
}

}  // namespace lbp
