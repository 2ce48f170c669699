// First convolution of the policy network (8x8 stride 4, C -> 32; Appendix F.1 / F.2) as a fused
// tcgen05 kernel: uint8 frames -> shared memory -> fp16 rows in tensor memory -> tensor cores.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include "common.cuh"

namespace hts {

struct Conv1Plan {
    int C, H, W;            // observation
    int Hs, Ws;             // space-to-depth(4) grid
    int H1, W1;             // conv1 output extent (Hs-1, Ws-1)
    int H1s, W1s, P1s;      // space-to-depth(2) grid of the output (input layout of conv2)
    int env_pitch;              // bytes of a box: what a staged entry holds of one environment
    int stage_bytes, stages;    // a staged entry, and how many of them shared memory holds for each of the kernel's two pipes
};

// Tensor maps over the caller's frame buffers, keyed by (address, frames): encoding one costs about a
// microsecond of host time and actor loops hand in the same few buffers again and again.
struct Conv1MapCache {
    static constexpr int kEntries = 16;
    const void* ptr[kEntries] = {};
    int frames[kEntries] = {};
    CUtensorMap map[kEntries];
    int next = 0;
};

// false if the geometry does not fit the kernel (C not 4, 8 or 16; H or W not a multiple of 4; too wide)
bool conv1_plan(const Geometry& g, Conv1Plan* plan);

// weight_map: w1 packed [128][16*C] fp16, scaled: row dy*64 + dx*32 + o, column c*16 + uy*4 + ux  holds  w1[o][c][4dy+uy][4dx+ux]
// out: fp16 rows [((y/2)*env_rows + env)*W1s + x/2][128], column ((y%2)*2 + x%2)*32 + o; env_rows: environments of the workspace
// ix: dense frames (row e = frame e of obs) or frames gathered by slot from a pool (see Indexing)
// dependent: the kernel loads the filter and biases before it waits for its predecessor, so it may start early only
// where that is not the one that packed them
hts_status conv1_launch(const Conv1Plan& pl, const CUtensorMap& weight_map, Conv1MapCache& maps, const uint8_t* obs,
                        const Indexing& ix, int n, const float* bias, const float* inv_scale, __half* out, int env_rows, int* status,
                        bool dependent, cudaStream_t s);

}  // namespace hts
