// Host-side helpers of the tensor-core kernels: tensor-map encoding through the driver entry
// point (looked up at run time, so the library does not link against libcuda).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace hts {
namespace tc {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// 2-D fp16 row-major [rows, cols] matrix, box [box_rows x 64 cols], 128-byte swizzle, zero fill.
inline bool make_map(CUtensorMap* m, const void* ptr, uint64_t rows, uint64_t cols, uint64_t pitch_bytes, uint32_t box_rows)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {pitch_bytes};
    const cuuint32_t box[2] = {64, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp16 rows of `channels` in the order (y, environment, x), seen as (channel, x, environment, y); box = 64 channels of one
// environment's grid, 128-byte swizzle.
inline bool make_grid_map(CUtensorMap* m, const void* ptr, int channels, int W, uint64_t envs, int H)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)channels * 2;
    const cuuint64_t dims[4] = {(cuuint64_t)channels, (cuuint64_t)W, envs, (cuuint64_t)H};
    const cuuint64_t strides[3] = {row, row * W, row * W * envs};
    const cuuint32_t box[4] = {64, (cuuint32_t)W, 1, (cuuint32_t)H};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// uint8 frames [frames, C, H, W] seen as 32-bit words [frames][C][H/4 grid rows][W words]: the four input
// rows under one grid row are W contiguous words.  Box = `group_rows` grid rows of `channels` channels of one frame.
inline bool make_frames_map(CUtensorMap* m, const void* ptr, int W, int H, int C, uint64_t frames, int group_rows, int channels)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)W, (cuuint64_t)(H / 4), (cuuint64_t)C, frames};
    const cuuint64_t strides[3] = {(cuuint64_t)4 * W, (cuuint64_t)H * W, (cuuint64_t)C * H * W};
    const cuuint32_t box[4] = {(cuuint32_t)W, (cuuint32_t)group_rows, (cuuint32_t)channels, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp32 row-major [rows, cols], box [box_rows x box_cols], no swizzle, zero fill.
inline bool make_f32_map(CUtensorMap* m, const float* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t box_cols)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * 4};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp32 activations seen as (x, row of a phase, phase, channel, frame); box = whole rows, `rows` of them in every phase of `channels`
// channels of one frame.
inline bool make_rows_map(CUtensorMap* m, const float* ptr, int pitch, int phase_rows, int phases, int C, uint64_t frames, int rows, int channels)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)pitch * 4, phase = row * phase_rows, chan = phase * phases;
    const cuuint64_t dims[5] = {(cuuint64_t)pitch, (cuuint64_t)phase_rows, (cuuint64_t)phases, (cuuint64_t)C, frames};
    const cuuint64_t strides[4] = {row, phase, chan, chan * C};
    const cuuint32_t box[5] = {(cuuint32_t)pitch, (cuuint32_t)rows, (cuuint32_t)phases, (cuuint32_t)channels, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, const_cast<float*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tc
}  // namespace hts
