// Internal declarations shared by the translation units of liblbp:
// host-side plan structures, launch prototypes and error plumbing.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

#include "lbp.h"

namespace lbp {

constexpr int kMaxOrder = 16;                    // largest WHT order k
constexpr int kMaxRank = kMaxOrder * kMaxOrder;  // r <= k*k

// Device status block at the start of every workspace (256 B reserved).
//   word 0: an lbp_status (LBP_ERR_TIMEOUT) written by a kernel whose wait expired
//   word 1: where that wait gave up (kernel id << 16 | site)
//   word 2: kStatusMagic, written together with word 0; the block counts as
//           "no error" unless the magic is present, so the caller's scratch
//           needs no initialisation.
constexpr size_t kStatusBytes = 256;
constexpr uint32_t kStatusMagic = 0x4C425045u;

// A validated basis list, prepared for the transform kernels.
//
// The kernels pool each k x k block down to LB x LB (LB = smallest power of two
// above the largest selected index; Walsh rows of sequency < LB are constant on
// runs of k/LB), run an LB x LB Hadamard butterfly in natural (Sylvester) order
// and pick the selected coefficients.  `qmap` maps a natural-order position
// (a, b) of that LB x LB array to the slot q of the basis list, -1 = unused.
struct BasisPlan {
  int32_t k;
  int32_t r;
  int32_t LB;
  int16_t qmap[kMaxRank];  // [a * LB + b]
  // order-k natural (Sylvester) row indices of the selected Walsh rows:
  // wal_{i_q}[u] = (-1)^popcount(nat_i[q] & u), likewise for j along W
  uint8_t nat_i[kMaxRank];
  uint8_t nat_j[kMaxRank];
  // the selected pairs themselves (sequency indices), slot by slot
  uint8_t seq_i[kMaxRank];
  uint8_t seq_j[kMaxRank];
};

// Validates (k, set, r) and fills `plan`.  Returns an lbp_status.
int make_basis_plan(int k, const lbp_basis* set, int r, BasisPlan* plan);

// Natural (Sylvester) row index of the length-n Walsh row with s sign changes.
int walsh_natural_index(int n, int s);
// wal_s[u] for order k: +1 or -1.
int walsh_sign(int k, int s, int u);

int check_order(int k);
// Blocks along a grid side of n tokens: sides that are not multiples of k are
// extended with zero tokens at their high end.
inline int blocks_along(int n, int k) { return (n + k - 1) / k; }

void set_last_cuda_error(cudaError_t e);
void count_launch(int n = 1);   // bumps the per-thread kernel-launch counter
void note_cuda_failure(cudaError_t e, const char* file, int line);   // LBP_VERBOSE_ERRORS=1: one line on stderr
#define LBP_CUDA_TRY(expr)                                 \
  do {                                                     \
    cudaError_t e__ = (expr);                              \
    if (e__ != cudaSuccess) {                              \
      ::lbp::set_last_cuda_error(e__);                     \
      ::lbp::note_cuda_failure(e__, __FILE__, __LINE__);   \
      return LBP_ERR_CUDA;                                 \
    }                                                      \
  } while (0)

// What is to be done once on each device, from whichever thread comes first (twice when two
// come at the same time, so it must bear that); on devices past the 63rd every time.
class PerDevice {
 public:
  template <class Action>
  int operator()(int dev, Action action) {
    const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
    if ((done_.load(std::memory_order_relaxed) & bit) != 0) return LBP_OK;
    if (int e = action()) return e;
    done_.fetch_or(bit, std::memory_order_relaxed);
    return LBP_OK;
  }

 private:
  std::atomic<uint64_t> done_{0};
};
// The opt-in to more than 48 KB of dynamic shared memory is a kernel's on one device.
inline int allow_dynamic_smem(PerDevice& per_device, const void* kernel, int bytes) {
  int dev = 0;
  LBP_CUDA_TRY(cudaGetDevice(&dev));
  return per_device(dev, [&]() -> int {
    LBP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    return LBP_OK;
  });
}

// ---- tensor maps (TMA descriptors), encoded on the host ------------------
// 4-D channels-last tensor (B, H, W, C): box = one k x k block x box_c
// channels; no swizzle, or the 128-byte swizzle (box_c * element size must be 128).
// `view`: strides of a tensor that is not dense (null, or all zero: dense).
int encode_block_tensor_map(CUtensorMap* map, const void* base, int dtype, int B, int H, int W,
                            int C, int k, int box_c, bool swizzle128,
                            const lbp_view* view = nullptr);
// Same tensor with an explicit box of box_h x box_w tokens.
int encode_box_tensor_map(CUtensorMap* map, const void* base, int dtype, int B, int H, int W, int C,
                          int box_c, int box_w, int box_h, bool swizzle128,
                          const lbp_view* view = nullptr);
// The strides a view stands for (dense when null or all zero).
inline lbp_view resolve_view(const lbp_view* v, int H, int W, int C) {
  if (v != nullptr && v->token != 0) return *v;
  return lbp_view{static_cast<int64_t>(H) * W * C, static_cast<int64_t>(W) * C, C};
}
inline bool is_dense(const lbp_view* v) { return v == nullptr || v->token == 0; }
// 2-D row-major bf16 matrix (rows, cols): box = box_rows x 64 columns (128 B),
// 128-byte swizzle.  pitch: elements between rows (0: dense).
int encode_matrix_tensor_map(CUtensorMap* map, const void* base, long long rows, long long cols,
                             int box_rows, long long pitch = 0);

// 2-D row-major fp32 matrix (rows, cols), no swizzle.
int encode_f32_matrix_map(CUtensorMap* map, const void* base, long long rows, long long cols, int box_rows,
                          int box_cols);

// ---- kernel launchers (each returns an lbp_status) ------------------------
// Row q of block blk of a projected tensor is row blk * r + q.
// `scale` multiplies the +-1 sums; 0 selects 1/k, the orthonormal coefficients of Eq. 6.
int launch_project(const void* t, void* t_hat, int dtype, int B, int H, int W, int C,
                   const BasisPlan& plan, uint32_t* status, cudaStream_t stream,
                   float scale = 0.f, const lbp_view* view = nullptr);

// Per-thread switch read by the projection launchers (umma::Params::defer_wait).
bool test_stall_projection();   // test hook (lbp_fused.cu)
void set_projection_defer_wait(bool on);
bool projection_defer_wait();

// Per-thread launch shape of the tensor-pipe projection kernels (set around a
// launch by the side-stream mode of lbp_backward_batch):
//   max_ctas      0 = one CTA per SM, else at most this many CTAs
//   whole_tpcs    launch the CTAs as clusters of two, so that they fill both SMs
//                 of a TPC and leave the other TPCs whole for the CTA pairs of a
//                 products kernel that runs beside them
//   programmatic  launch with programmatic stream serialization
struct ProjLaunch {
  int max_ctas;
  bool whole_tpcs;
  bool programmatic;
};
void set_projection_launch(ProjLaunch shape);
ProjLaunch projection_launch();

// Projects two tensors that share the token grid (x and g_y) in one launch.
int launch_project2(const void* t0, void* out0, int C0, const void* t1, void* out1, int C1,
                    int dtype, int B, int H, int W, const BasisPlan& plan,
                    uint32_t* status, cudaStream_t stream, float scale0 = 0.f, float scale1 = 0.f,
                    const lbp_view* view0 = nullptr, const lbp_view* view1 = nullptr);

// One-pass spectrum (bf16 data, k = 4 or 8): energy[i*k + j] of all k*k responses.
// plan: all k*k pairs in raster order.
bool spectrum_mma_supported(int k, int dtype);
int launch_spectrum_mma(const void* t, int B, int H, int W, int C, const BasisPlan& plan,
                        double* energy, uint32_t* status, cudaStream_t stream);

// energy[q] (device, r doubles, overwritten) = sum of squares of the rows
// q, q + r, ... of t_hat (rows x C of `dtype`).
int launch_square_reduce(const void* t_hat, int dtype, long long rows, int C, int r, double* energy,
                         cudaStream_t stream);

// t_hat is fp32 when `in_f32`, else of `dtype`; t is of `dtype`.
int launch_expand(const void* t_hat, bool in_f32, void* t, int dtype, int B, int H, int W, int C,
                  const BasisPlan& plan, cudaStream_t stream,
                  const lbp_view* view = nullptr);

// D[M, N] = sum_k A(m, k) * B(k, n), fp32 accumulation.
//   a_mn_major == false: A is stored (M, K) row-major;  true: A is stored (K, M) row-major.
//   B is stored (K, N) row-major.  D is (M, N) row-major of d_dtype.
// bf16 operands run on tcgen05 tensor cores; fp32 operands on FFMA.
// `splitk_ws` holds fp32 partial tiles when the kernel splits K.
int launch_gemm(const void* A, bool a_mn_major, const void* Bm, void* D, int in_dtype, int d_dtype,
                long long M, long long N, long long K, float* splitk_ws, size_t splitk_ws_bytes,
                uint32_t* status, cudaStream_t stream);
// fp32 products (gemm_fp32.cu): one or two independent ones in one launch; M (when
// a_mn), K (when not) and N are multiples of 4, operands 16-byte aligned.
struct GemmFp32 {
  const float *A, *B;
  float* D;
  long long M, N, K;
  bool a_mn;
};
int launch_gemm_fp32(const GemmFp32* jobs, int n, float* ws, size_t ws_bytes, uint32_t* status, cudaStream_t stream);
// Scratch for the K slices these take at best (with less, K is sliced less or not at all).
size_t gemm_fp32_ws_bytes(const GemmFp32* jobs, int n);
void set_test_stall_fp32(bool on);   // test hook (gemm_fp32_split.cu)
void gemm_fp32_plan(const GemmFp32 (&jobs)[2], size_t room, int64_t* out6);   // test hook
size_t gemm_splitk_ws_bytes(long long M, long long N, long long K, int in_dtype);
// D[i] = beta * D[i] + sum over `splits` fp32 planes of mn elements each (mn a multiple
// of 4), in plane order; D is not read when beta is 0.  `late`: the next kernel on the
// stream is one of many small CTAs (which would all settle on the SMs that are idle if they
// came early), not one of a CTA per SM.
int launch_splitk_reduce(const float* planes, void* D, long long mn, int splits, bool d_bf16,
                         float beta, bool late, cudaStream_t stream);

int check_device_arch();

// ---- kernels around Algorithm 1 (lbp_extras.cu) ----
// g_W <- beta * g_W + a (+ b); a, b fp32 of mn elements, g_W fp32 or bf16.
int launch_gw_combine(void* g_W, bool gw_bf16, const float* a, const float* b, float beta,
                      long long mn, cudaStream_t stream);
// Where token i of a tensor of HW-token images (rows of W tokens) starts, in
// the units of the strides: (i / HW) * s_image + ((i % HW) / W) * s_row + (i % W) * s_tok.
// Rows with a pitch: HW = W = 1, s_image = pitch.
struct TokenMap {
  int32_t HW, W;
  long long s_image, s_row, s_tok;
  __host__ __device__ long long offset(long long i) const {
    // (a 64-bit division costs a kernel more than what it addresses)
    const long long b = i < (1ll << 31) ? static_cast<int>(i) / HW : i / HW;
    const int t = static_cast<int>(i - b * HW);
    return b * s_image + (t / W) * s_row + (t % W) * s_tok;
  }
};
inline TokenMap token_map(const lbp_view& v, int H, int W) {
  return TokenMap{H * W, W, v.image, v.row, v.token};
}
// Gathers (to_dense) or scatters n_tok tokens of C channels between a tensor
// laid out as `tm` says (element strides, multiples of 16 bytes) and a dense
// (n_tok, C) matrix.
int launch_copy_tokens(const void* src, void* dst, bool to_dense, long long n_tok, int C, int dtype,
                       TokenMap tm, cudaStream_t stream);
// g_bias <- beta * g_bias + scale * (sum of n_a rows of a) + (sum of n_b rows of b), fp64
// sums.  r > 0: the rows of a are the coefficients of slot q of its blocks (dense, r
// per block); r == 0: tokens under `ta`.  b: tokens under `tb`.  g_bias is fp32 or bf16.
// scratch: for the sums of parts of the rows, as many as fit.
int launch_bias_grad(const void* a, long long n_a, int r, int q, TokenMap ta, double scale,
                     const void* b, long long n_b, TokenMap tb, int C, int dtype, void* g_bias,
                     bool out_bf16, float beta, double* scratch, size_t scratch_bytes, cudaStream_t stream);

// Tuning switches, read from the environment once (first use):
//   LBP_FUSED=0          separate product and expansion kernels instead of the
//                        persistent products kernel
//   LBP_PAIR=0           one-CTA products kernel also on wide layers
//   LBP_PROJECT_UMMA=0   bf16 projection by additions on the CUDA cores instead of tcgen05
//   LBP_FUSED_TILES=a,b,c  column tiles of the two products and K slices of g_W
//   LBP_FP32_FORM=n      fp32 products: 0 on FFMA, 1 / 2 split operands on tcgen05 in tiles
//                        of 128 x 64 / 128 x 128 (unset or anything else = chosen by size);
//                        n,p: in items of p k-blocks, where the workspace has room
//   LBP_FUSED_VERBOSE=1  print the chosen tile plan
//   LBP_BATCH_PROJ_SMS=n lbp_backward_batch: SMs given to the projection of the next
//                        layer while the products kernel of a layer runs (0 = one
//                        kernel at a time; unset = chosen per pair of layers)
//   LBP_BATCH_ORDER=a,b,.. lbp_backward_batch (up to 6 problems): the order in which
//                        the problems are taken (read at every call)
struct TuneOptions {
  bool fused, pair, umma, verbose, has_tiles;
  int tiles_bnw, tiles_bnx, tiles_splits;
  int batch_proj_sms;   // -1 = library default
  int fp32_form;        // -1 = chosen by size
  int fp32_per;         // 0 = chosen by size
};
const TuneOptions& tune_options();
void reload_tune_options();   // test hook: read the environment again

// Every host-side check of one lbp_backward call (pointers, layer, basis list,
// alignment, workspace size); nothing is enqueued.  Returns an lbp_status.
int validate_backward_call(const void* x, const void* g_y, const void* W, const void* g_x,
                           const void* g_W, const lbp_layer* layer, const lbp_basis* set, int r,
                           const void* ws, size_t ws_bytes);

}  // namespace lbp
