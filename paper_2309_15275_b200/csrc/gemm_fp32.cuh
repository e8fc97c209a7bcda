// Shared by the two kernels of the fp32 products (FFMA and split operands on tcgen05).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbp {

// A product as its kernel sees it: tiles of D, each over K in `chunks` items of at most
// `per` k-blocks.
struct GemmFp32Job {
  const float *A, *B;
  float* D;                       // chunks > 1: the planes [chunks][M][N]
  long long M, N, K;
  int32_t a_mn, tiles_c, tiles;   // tiles of D along its columns (FFMA: N; split: the operand not in TMEM), in all
  int32_t kb, per, chunks;        // k-blocks; of an item; items per tile
};
struct GemmFp32Jobs {
  GemmFp32Job j[2];
  int32_t items0, items;          // items of the first job, of both
  uint32_t* status;
  int32_t test_stall;             // failure injection (lbp_test_stall_products): no loads
};

// n: one job or two; bn: columns of a tile, 64 or 128.
int launch_gemm_fp32_split(GemmFp32Jobs& js, int n, int bn, cudaStream_t stream);

}  // namespace lbp
