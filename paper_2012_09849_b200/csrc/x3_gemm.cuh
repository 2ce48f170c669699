// fp32-accurate contractions on the tensor cores ("x3": every fp32 operand as three bf16 pieces).
//
// A fp32 number is the exact sum of three bf16 numbers (3 x 8 significant bits; the pieces are the successive
// round-to-nearest remainders).  A product of two such sums has nine terms; the six whose weight is at least
// 2^-16 of the leading one are multiplied by tcgen05.mma (bf16 products are exact, accumulation is fp32) and the
// three below 2^-24 are dropped: less than one rounding of an fp32 multiply-add.  The terms of weight 1, 2^-8 and
// 2^-16 go to accumulators of their own, which are added smallest first.
//
// Accumulation.  The tensor core does not round a sum to nearest but cuts it off: a chain of s instructions (16 products
// each) comes out too small by up to s last places, s / 2 on average, all in one direction.  So a chain is eight
// instructions, 128 of K, and the epilogue warps add the chains in registers, rounded to nearest, while the next ones
// run.  Error (2-norm against 64 bits, learner batches of 5 to 1024 of four frame shapes), conv1's weights and the
// whole gradient: one chain per tile or range of rows (16 to 200 instructions) 5 to 33e-7 and 2 to 13e-7, fp32
// multiply-adds in order 2 to 11e-7 and 2 to 10e-7, chains of eight 2 to 6e-7 and 1 to 10e-7 (what is left is the forward
// pass and the heads).  Chains of four are no closer and take 4 % longer; eight cost 2 % of a gradient of 1024 (860 to 876 us).
//
// Layouts: activations and gradients are stored as three planes of pixel-major rows [rows][channels] bf16, so
// that the data gradient of a convolution is a sum over taps of row-shifted products on a flat pixel grid (x3_dgrad)
// and its weight gradient one contraction over the rows per tap (x3_wgrad).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include "common.cuh"

namespace hts {

// ---- data gradients: D[m, n] = sum over (chunk, tap) of A[m + shift(tap), chunk] . B[n, tap, chunk] -------------
enum X3Mode {
    X3_DGRAD_FC,            // gradient of conv3's output: N tile = pixel, planes on conv3's input grid
    X3_DGRAD,               // gradient of conv2's output: planes on conv2's input grid
    X3_DGRAD_S2D            // gradient of conv1's output: N tile = row parity, planes interleaved in 128-column rows
};

struct X3TapParams {
    int mode;
    int m_tiles, n_tiles;               // work: m_tiles x n_tiles tiles of 128 rows x 64 columns
    int chunks;                         // 64-row K chunks of the packed weights
    int taps, tpe;                      // filter taps; taps served by one A entry (taps, or 1 for very wide grids)
    int shift[9], lo;                   // row shift of each tap, and the smallest
    int entry_rows;                     // rows of an A entry: 128 + spread of the shifts, or 128
    int entries, b_stages;              // ring sizes
    int tap_cols;                       // columns of the packed weights per tap
    int n;                              // observations
    int P, W;                           // grid of the rows m: positions per observation, width
    int H_out, W_out;                   // valid extent
    int P_dst, W_dst, dst_pitch;        // destination grid, elements per row
    size_t dst_plane;                   // elements between planes
    __nv_bfloat16* dst;
    const __nv_bfloat16* mask;          // first plane of the activation whose ReLU the gradient passes, [m][mask_pitch]
    int mask_pitch;
    int* status;
};

// b: the forward pass's packed weights (K, the layer's outputs, along the rows: no transposed copy is kept)
hts_status x3_dgrad_launch(const CUtensorMap& a, const CUtensorMap& b, const X3TapParams& p, cudaStream_t s);
// Fills taps / tpe / shift / lo / entry_rows / ring sizes; false if nothing fits.
bool x3_taps_plan(X3TapParams* p, int chunks, int taps, const int* shift);

// ---- partial weight gradients: D[m, n] = sum over a range of rows k of A[k + shift, m] . B[k, n] ---------------
// A CTA (kind, range) loads A slabs (64 columns x rows, all planes) and B slabs per stage of `kr` rows and forms up
// to two groups of 128 x NB: a group's M = two 64-column blocks at a_off and a_off + lbo (two taps of one slab, or
// two slabs).
constexpr int kX3MaxSlabs = 16, kX3MaxGroups = 32;
template <int NB> constexpr int kX3StageRows = NB == 64 ? 64 : 128;
struct X3WgradParams {
    int kr, stages;                     // rows per stage (kX3StageRows), stages in the ring
    int a_rows;                         // rows of an A slab (kr + spread of the taps)
    int n_a, n_b;                       // slabs per stage
    int ka, a_step, b_step;             // columns: A (kind % ka) * a_step + slab_col, B (kind / ka) * b_step + 64 * slab
    int slab_mul, slab_col[kX3MaxSlabs], slab_row[kX3MaxSlabs];   // of slab kind * slab_mul + s
    int group_mul, groups, group_cap;   // group index = kind * group_mul + g, g < groups; indices >= group_cap are skipped
    int a_off[kX3MaxGroups], a_lbo[kX3MaxGroups];   // by group index
    int b_off[2];                       // by g
    int kinds, last_ranges, ranges;     // ranges per kind (the last kind has its own count)
    int row_chunks;                     // chunks of kr rows in total
    float* part;                        // [group index][range][128][NB], or nullptr
    size_t group_stride;                // floats between group indices
    float* bias_part;                   // [range][NB], written by kind 0, or nullptr
    float* fc_w;                        // dense gradient [512][pixel * 64 + c], or nullptr
    int P3;
    int* status;
};
// A data gradient on d_blocks blocks and, beside it, a weight gradient that does not need it.
hts_status x3_data_weights_launch(const CUtensorMap& da, const CUtensorMap& db, const X3TapParams& d, int d_blocks, const CUtensorMap& wa,
                                  const CUtensorMap& wb, const X3WgradParams& w, cudaStream_t s);
// The weight gradients of the second and the first convolution side by side.
hts_status x3_weights_launch(const CUtensorMap& a2, const CUtensorMap& b2, const X3WgradParams& w2, const CUtensorMap& a1, const CUtensorMap& b1,
                             const X3WgradParams& w1, cudaStream_t s);

// bf16 [planes][rows][cols], box 64 columns x box_rows x box_planes, 128-byte swizzle, zero fill
bool x3_make_map(CUtensorMap* m, const void* ptr, uint64_t cols, uint64_t rows, uint64_t planes, uint64_t pitch_elems,
                 uint64_t plane_elems, uint32_t box_rows, uint32_t box_planes);

#ifdef __CUDACC__
// Two fp32 values -> three packed bf16 pairs whose sums are the values.  Where a first piece is infinite (a magnitude
// above 3.39e38 rounds to that too) the lower ones mean nothing, or are zero with ZERO_LOW: a sum of first pieces, or of
// products of first pieces, that is not finite is the value by itself (x3_sum), so that a sum is infinite or NaN where
// its fp32 form is.  The frames' gradient has one finite piece on its other side: zero lower pieces are enough there.
template <bool ZERO_LOW = false>
__device__ __forceinline__ void x3_split2(float a, float b, uint32_t& p0, uint32_t& p1, uint32_t& p2)
{
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p0) : "f"(b), "f"(a));
    const float ha = __uint_as_float(p0 << 16), hb = __uint_as_float(p0 & 0xffff0000u);
    const float ra = !ZERO_LOW || fabsf(ha) < INFINITY ? a - ha : 0.f, rb = !ZERO_LOW || fabsf(hb) < INFINITY ? b - hb : 0.f;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p1) : "f"(rb), "f"(ra));
    const float sa = ra - __uint_as_float(p1 << 16), sb = rb - __uint_as_float(p1 & 0xffff0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p2) : "f"(sb), "f"(sa));
}
// A sum of first pieces (or of products of them) and what the lower ones add to it.
__device__ __forceinline__ float x3_sum(float first, float low) { return first + (fabsf(first) < INFINITY ? low : 0.f); }
#endif

}  // namespace hts
