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
// fill.  The frames that fit have P1s + P2 from 71 to 208.  Measured, frames not in cache, here / there, us per step:
//   per SM             3             4             5             6
//   88 x 36  (71)    24.3 / 24.4   27.7 / 25.6
//   60 x 60  (85)    24.6 / 25.2   29.7 / 28.2
//   44 x 96  (100)   24.7 / 25.2   29.8 / 28.7
//   72 x 72  (130)   26.9 / 27.3   30.6 / 29.2
//   76 x 76  (145)   27.5 / 28.8   31.3 / 31.4   35.4 / 33.5
//   64 x 96  (156)   27.0 / 27.8   32.0 / 32.2   36.2 / 34.0
//   84 x 84  (181)   28.6 / 31.1   32.7 / 33.1   38.4 / 38.7   42.5 / 41.3
//   100 x 80 (208)   31.3 / 33.9   35.7 / 37.1   40.4 / 40.9   44.9 / 44.2
// Frames with a conv1 tile more than others of their size lie one step too high: 60 x 72 (105) 26.4 / 25.9 at three, 80 x 80 (164)
// 32.7 / 31.7 at four, 120 x 60 (183) 40.1 / 39.7 at five.
inline int conv_stack_envs(const ConvStackParams& p)
{
    const int per_sm = (p.P1s + p.P2) / 36;
    return per_sm < 3 ? 3 : per_sm;
}
// Weight maps: the packed filters of conv1 [128][64], conv2 [64][512] and conv3 [64][576], box 64 x 64.
// t1, t2: where conv1's and conv2's outputs go, as (channel, x, environment, y), box 64 channels x one environment's grid.
// dependent: as in conv1_launch.
hts_status conv_stack_launch(const CUtensorMap& w1, const CUtensorMap& w2, const CUtensorMap& w3, const CUtensorMap& t1, const CUtensorMap& t2,
                             const ConvStackParams& p, bool dependent, cudaStream_t s);

}  // namespace hts
