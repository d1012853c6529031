// npp_gemm.cuh -- BF16 tensor-core GEMM (tcgen05 + TMA).
//
//   C[m][n] = sum_k A[m][k] B[n][k]      A: M x K, B: N x K, both BF16 with K
//                                        contiguous ("K-major"), FP32 sums
//
// M a multiple of 128, N of the tile width BN (128 or 256), K of 64.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "npp_tcgen05.cuh"

namespace npp {

// C [M][N] = A B^T in tiles bn columns wide; ta boxes of 128 rows, tb boxes
// of box_b rows: bn, or 128 with bn = 256 where gemm_pairs (CTA pairs, each
// CTA loading half of B's rows).  *err is set nonzero if a pipeline wait
// timed out.
bool gemm_pairs(int M, int N);
cudaError_t launch_gemm(const CUtensorMap& ta, const CUtensorMap& tb, int M, int N, int K, int bn, int box_b, float* C,
                        int* err, cudaStream_t s);

}  // namespace npp
