// npp_mlp.cuh -- the sampling-proposal network's forward and backward passes
// as fused tensor-core kernels (npp_mlp.cu).
//
// Network: 72 inputs (padded to 128) -> 256 -> 256 -> 900 outputs: the 450
// parameters' means, then their log-standard-deviations (padded to D3 =
// 1024 rows).  The forward pass reads W3 in an order of its own: tiles of 256
// rows, 128 means and the same parameters' 128 log-stds (mlp_row), so that a
// tile's accumulator holds both outputs of a parameter.  Batches are rounded
// up to whole tiles of 128 rows.
#pragma once

#include <cstdint>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/npp_proposal.h"

namespace npp {

constexpr int MLP_NIN = NPP_PROP_NIN;      // 72
constexpr int MLP_D0 = 128;                // padded input width
constexpr int MLP_HID = NPP_PROP_HIDDEN;   // 256
constexpr int MLP_NTH = NPP_PROP_NTHETA;   // 450
constexpr int MLP_D3 = 1024;               // padded output width
constexpr int MLP_TP = 128;                // parameters per output tile

// row of the forward pass's W3 that holds output o (mean of parameter o, or
// log-std of parameter o - 450)
__host__ __device__ constexpr int mlp_row(int o)
{
    const int i = o < MLP_NTH ? o : o - MLP_NTH;
    return (i / MLP_TP) * 2 * MLP_TP + (o < MLP_NTH ? 0 : MLP_TP) + i % MLP_TP;
}

struct MlpForward {
    const float* x;            // [n][72]
    int n;                     // rows
    const float *b1, *b2, *b3; // biases [256], [256], [1024]
    float ls_min, ls_max;
    int groups;                // CTAs' shares of the four output tiles: 1, 2 or 4 per row tile
    int* err;                  // set nonzero when a pipeline wait timed out
    // inference: mean and std [n][450]
    float *mean, *sd;
    // training (theta set): activations for the backward pass and the loss
    const float* theta;        // [n][450]
    __nv_bfloat16 *X, *dY;     // [n][128], [n][1024] (H1, H2 [n][256] through their tensor maps)
    uint4* mask;               // [2 layers][n][2] bits of the positive activations
    float* loss_part;          // [n/128][4 tiles][8 warps]
};

struct MlpBackward {
    int n;
    const uint4* mask;         // as MlpForward::mask
    int* err;
};

// weight gradients dW3 [1024][256], dW2 [256][256], dW1 [256][128], the batch
// of product k split into splits[k] slices, each slice's partial sums written
// to part[k] + z size[k]
struct MlpGrads {
    int n;
    int splits[3];
    float* part[3];
    int* err;
};

// operands in blocks of 64 columns: the weights' boxes 256 rows, H1 and H2 128
struct MlpForwardMaps {
    CUtensorMap w1, w2, w3, h1, h2;
};
cudaError_t launch_mlp_forward(const MlpForwardMaps& m, const MlpForward& f, cudaStream_t s);
// dY, dZ2, dZ1 in boxes of 128 rows, W3 and W2 of 64
struct MlpBackwardMaps {
    CUtensorMap dy, w3, w2, dz2, dz1;
};
cudaError_t launch_mlp_backward(const MlpBackwardMaps& m, const MlpBackward& b, cudaStream_t s);
// the six operands in 64 x 64 boxes: dY, H2, dZ2, H1, dZ1, X
struct MlpGradMaps {
    CUtensorMap a[3], b[3];
};
cudaError_t launch_mlp_grads(const MlpGradMaps& m, const MlpGrads& g, cudaStream_t s);

// CTA shares of the output tiles for n rows: as many as keep the CTAs within
// one wave of the SMs
int mlp_groups(int n, int sms);
// batch slices of the weight gradients
void mlp_grad_splits(int n, int splits[3]);
int mlp_sm_count();

}  // namespace npp
