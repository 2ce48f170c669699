// fp32 convolutions of the actor step in strips: a thread owns PX consecutive pixels of one output row and OT channels.
#pragma once
#include <cuda.h>
#include "common.cuh"

namespace hts {

// One convolution of the fp32 path, whichever kernel computes it.
struct ConvParams {
    const void* x;                      // [frames][C][rows], u8 or fp32
    const float *w, *b;                 // [O][C k k], [O]
    const float* wk;                    // the same weights as [C k k][O], 16-byte aligned, or nullptr
    float* y;                           // [n][O][rows]
    int n, C, H, W, O, k, s, Ho, Wo;
    RowLayout xl, yl;
    float in_scale;
    int frame0;                         // fp32: frame of the layer's map that is x
    const int32_t* slots;               // frame of each row, or nullptr
    int pool;
    int* status;
    bool w_vec, words;                  // weights 16-byte aligned; frames 4-byte aligned
    bool y_rows;                        // outputs (or planes) are not one dense run of pixels per channel: a pixel's row is needed
    __nv_bfloat16* planes;              // optional second output: three bf16 planes of pixel-major rows (x3_gemm.cuh)
    size_t plane;
    int W_rows, P_rows;                 // its grid; 2 x 2 pixels per row when s2d
    bool s2d;
    bool early;                         // the next kernel is beside_conv1: its blocks may settle while the last ones of this run
};

#ifdef __CUDACC__
// Frame of batch row e: e itself, or its slot in the pool (a slot outside it is reported and reads frame 0).
__device__ __forceinline__ size_t frame_of(const ConvParams& p, int e)
{
    if (!p.slots) return (size_t)e;
    const int sl = p.slots[e];
    if ((unsigned)sl >= (unsigned)p.pool) { atomicCAS(p.status, 0, kStatusBadSlot); return 0; }
    return (size_t)sl;
}
// Where the inputs of output row i start, and its filter row u relative to that; where output row i is.  Divisions by one or two
// phases as shifts: a tile's block does them for every input that it looks up (step of one 84 x 84 x 4 frame that allocates nothing 47.3 us
// with divisions, 45.3).
__device__ __forceinline__ int x_row(const ConvParams& p, int i) { return i * (p.s >> (p.xl.phases - 1)) * p.xl.pitch; }
__device__ __forceinline__ int row_at(const RowLayout& l, int y) { return (y & (l.phases - 1)) * l.phase + (y >> (l.phases - 1)) * l.pitch; }
__device__ __forceinline__ int x_tap(const ConvParams& p, int u) { return row_at(p.xl, u); }
__device__ __forceinline__ int y_row(const ConvParams& p, int i) { return row_at(p.yl, i); }
// Where pixel (i, x) of row e starts in the planes.
__device__ __forceinline__ size_t plane_row(const ConvParams& p, int e, int i, int x)
{
    return p.s2d ? ((size_t)e * p.P_rows + (size_t)(i >> 1) * p.W_rows + (x >> 1)) * 128 + ((i & 1) * 2 + (x & 1)) * 32
                 : ((size_t)e * p.P_rows + i * p.Wo + x) * 64;
}
#endif

// Tiles of px pixels x oc channels that the fullest SM has (policy_ref.cu), and whether large ones are the faster tiles: one of 128 x 64
// (256 x 32) costs as much as 2.5 of 64 x 32 and 0.7 more for its start.
inline long conv_tiles(const ConvParams& p, int px, int oc)
{
    const long tiles = (long)(((size_t)p.n * p.Ho * p.Wo + px - 1) / px) * (p.O / oc), sms = device_sm_count(device_slot());
    return (tiles + sms - 1) / sms;
}
inline long conv_large_tiles(const ConvParams& p) { return p.O == 64 ? conv_tiles(p, 128, 64) : conv_tiles(p, 256, 32); }
inline bool conv_tiles_large(const ConvParams& p) { return 2 * conv_tiles(p, 64, 32) > 5 * conv_large_tiles(p) + 1; }

// Boxes of a context's activations, as the forms of the second and third layer read them.
struct StripMaps { CUtensorMap few2, thin2, some2, many2, few3, thin3, some3; };
bool make_strip_maps(const Geometry& g, const RefWorkspace& ws, size_t frames, StripMaps* maps);

// HTS_ERR_UNSUPPORTED: not a shape for strips (nothing was launched).
hts_status launch_conv_strip(const ConvParams& p, const StripMaps* maps, cudaStream_t s);

}  // namespace hts
