// fp32 dense layer of the actor step for batches that fill the device.
#pragma once
#include <cuda.h>
#include "common.cuh"

namespace hts {

// h[e,o] = relu(b[o] + the 32 chains f = l, l + 32, ... of x[e,f] w[o,f], added as a binary tree over l (halves first)).
// F is a multiple of 64.
struct FcParams {
    const float* b;                     // [512]
    float* h;                           // [n][512]
    int n, F, row0;                     // row0: row of x's map that is the batch's first
    int* status;
};
constexpr int kFcBoxRows = 16, kFcBoxCols = 128;
struct FcMaps { CUtensorMap x, w; bool ok; };   // boxes of x [frames][F] and w [512][F]; ok: they were made
// false: the driver refused.  Not made for fewer columns than a box has.
bool make_fc_maps(const float* x, const float* w, int F, size_t frames, FcMaps* m);

// HTS_ERR_UNSUPPORTED: no maps (nothing was launched).
hts_status launch_fc_lanes(const FcParams& p, const FcMaps& m, cudaStream_t s);

}  // namespace hts
