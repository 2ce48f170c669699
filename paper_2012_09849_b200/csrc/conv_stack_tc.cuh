// The three convolutions of the policy network (Appendix F.1 / F.2) in one kernel for four-channel frames.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include "common.cuh"

namespace hts {

struct ConvStackParams {
    const uint8_t* obs;
    const int32_t* slots;               // frame of each row in obs, or nullptr: row e is frame e
    int pool;                           // frames in obs when slots are given
    int n;
    int row0;                           // the batch's first row of the workspaces
    int H, W, Ws;                       // frame, and width of its space-to-depth(4) grid
    int H1, W1, W1s, P1s;               // conv1 output; width and positions of its space-to-depth(2) grid
    int H2, W2, P2, H3, W3, P3;
    int tiles;                          // conv1 tiles of 124 grid positions per environment
    int a1_plane, a2_bytes, raw_bytes;  // shared memory: one 64-channel plane of conv1's output, conv2's output, one frame
    const float *b1, *b2, *b3;
    const float *inv1, *inv2, *inv3;    // device scalars undoing the weight scaling (and conv1's /255)
    __half* a3;                         // the dense layer's input
    int* status;
};

// false if the frames do not fit the kernel (four channels; one 128-row tile must hold conv2's and conv3's grids)
bool conv_stack_plan(const Geometry& g, ConvStackParams* p);
// Batches up to this many environments per SM are faster here than in a kernel per layer.  A kernel per layer fills its tiles
// from several environments; here an environment's conv2 and conv3 take a tile of 128 rows each, however few of them its grids
// fill.  Measured, here / there, us per step: 84 x 84 (100 and 81 rows) 33.2 / 33.9 at four per SM, 38.4 / 39.3 at five, 42.6 /
// 42.1 at six; 64 x 96 (96 and 60 rows) 32.5 / 32.7 at four, 36.6 / 34.6 at five.
inline int conv_stack_envs(const ConvStackParams& p)
{
    const int per_sm = (p.P1s + p.P2) / 36;
    return per_sm < 2 ? 2 : per_sm < 6 ? per_sm : 6;
}
// Weight maps: the packed filters of conv1 [128][64], conv2 [64][512] and conv3 [64][576], box 64 x 64.
// t1, t2: where conv1's and conv2's outputs go, as (channel, x, environment, y), box 64 channels x one environment's grid.
// dependent: as in conv1_launch.
hts_status conv_stack_launch(const CUtensorMap& w1, const CUtensorMap& w2, const CUtensorMap& w3, const CUtensorMap& t1, const CUtensorMap& t2,
                             const ConvStackParams& p, bool dependent, cudaStream_t s);

}  // namespace hts
