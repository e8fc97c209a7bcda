// Shared between the two projection kernels (additions-only and tensor-pipe).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "lbp_internal.h"

namespace lbp {

// One launch projects up to two tensors that share the token grid (x and g_y of
// a layer): items [0, n_items0) belong to tensor 0, the rest to tensor 1.
struct ProjParams {
  int32_t nb, Hb, Wb, r;
  int32_t C[2], n_chunks[2];
  uint32_t n_items0, n_items;   // nb * n_chunks[0], nb * (n_chunks[0] + n_chunks[1])
  uint32_t* status;
  // factor applied to the +-1 sums of tensor 0 / 1: 1/k gives the orthonormal
  // coefficients of Eq. 6; the products kernel asks for other powers of two
  float scale[2];
};

template <int K, bool BF16>
struct ProjCfg {
  static constexpr int kTileBytesMax = K * K * 128;
  static constexpr int kWarps = (K == 16) ? 6 : 12;
  static constexpr int kStages = (K == 4) ? 4 : (K == 8 ? 2 : 1);
  static constexpr int kSmemBytes = kWarps * kStages * kTileBytesMax + kWarps * kStages * 8 + 128;
};

// tcgen05 tensor cores (bf16): orders 8 and 16 at r <= 48, order 4 at every rank.
// Coefficients are written densely (block blk: rows blk * r ..); t1 may be null.
bool project_umma_supported(int k, int r);
int launch_project_umma(const void* t0, void* out0, int C0, const lbp_view* view0, const void* t1,
                        void* out1, int C1, const lbp_view* view1, int B, int H, int W,
                        const BasisPlan& bp, float scale0, float scale1, int sms, uint32_t* status,
                        cudaStream_t stream);

}  // namespace lbp
