// The dense layer (F -> 512) of the policy network on pairs of SMs (Appendix F.1 / F.2).
#pragma once
#include <cuda.h>
#include "common.cuh"

namespace hts {

struct FcPairParams {
    int splits, cps;                    // K ranges, 64-column chunks of a range
    int group;                          // ranges of one pair of SMs (the last pair of a tile may have fewer)
    int n;                              // valid rows
    int row0;                           // the first one's row of the activations
    const float* bias;                  // [512]
    const float* inv_scale;             // device scalar undoing the weight scaling
    float* h;                           // [n][512]: written where one pair has all ranges
    float* planes;                      // otherwise [plane][rows][512]: the sum of the first pair's ranges, then one per further range
    size_t plane_stride;
    int* status;
};

// Ranges of a pair, and with it the planes left to add up (1: the hidden layer itself), for n rows on a device.
struct FcPairPlan {
    bool wide;                          // 256 x 256 tiles, else 256 x 128
    int group, planes;
};
FcPairPlan fc_pair_plan(int n, int splits);
// act_map: [rows][F], box 128 x 64.  weight_map: [512][F], box 64 x 64.
hts_status fc_pair_launch(const CUtensorMap& act_map, const CUtensorMap& weight_map, const FcPairParams& p, bool wide, cudaStream_t s);

}  // namespace hts
