// Stride-1 convolution with its filter resident in shared memory, marching down the rows of a pixel grid: the second and
// third convolutions of the policy network (Appendix F.1 / F.2).
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include "common.cuh"

namespace hts {

struct ConvRowsParams {
    int n_env;              // valid environments
    int W_in;               // input grid: width
    int H_out, W_out;
    int in_plane;           // input rows of one grid row: environments of the workspace x W_in
    int tiles;              // 128-column tiles of n_env * W_in
    int col0;               // the batch's first column (environment, x)
    const float* bias;      // [64]
    const float* inv_scale; // device scalar undoing the weight scaling
    __half* out;            // [64] per output pixel, at env * out_env + y * out_y + x * 64
    size_t out_env, out_y;
    int* status;
};

// KY x KX filter taps over CPT planes of 64 channels: (2, 2, 2) for conv2 on the space-to-depth grid, (3, 3, 1) for conv3.
// Rows of the input matrix are (y, environment, x); act_map's box is kConvRowsBox<KX> of them x 64 channels.  weight_map:
// [64][(dy, dx, plane) x 64], box 64 x 64.
template <int KX> constexpr int kConvRowsBox = 128 + KX - 1;
template <int KY, int KX, int CPT>
hts_status conv_rows_launch(const CUtensorMap& act_map, const CUtensorMap& weight_map, const ConvRowsParams& p, cudaStream_t s);

}  // namespace hts
