// conv1 (8x8/4, 4 -> 32), conv2 (4x4/2 -> 64) and conv3 (3x3/1 -> 64) from raw frames to the dense layer's input, one
// environment at a time per CTA with every filter resident in shared memory (152 KB).
//
// For batches of a few environments per SM, where three kernels spend their time between them: each starts 1.3 us after
// the last CTA of the one before and needs 2 us to its first finished tile.  Step of 16 observations: 20.5 -> 16.9 us, of 256: 27.3
// -> 24.5, of 444: 31.6 -> 29.1; at five environments per SM they are equal (conv_stack_envs).  From there on the three
// kernels win: one environment here takes about 7800 clocks where its MMAs need 4288,
// because those fetch their operands from the same shared memory (128 bytes per clock, 68 x 6 KB per environment) that the
// converters and epilogues work in.  The activations never leave the SM between layers: a CTA keeps one frame (raw bytes), conv1's output (K-major 128-byte-swizzled rows, two
// planes of 64 channels of the space-to-depth(2) grid) and conv2's output (one plane) in shared memory, and
// consecutive environments overlap, conv1 of the next one running under conv2 and conv3 of this one.
//
//   * conv1 is a 2x2/1 convolution on the space-to-depth(4) grid, flat position q = Y * Ws + X.  A tile is 124
//     positions; the operand of the two filter rows (positions q and q + Ws) is converted from bytes in registers (a
//     zero-extended byte is the fp16 subnormal b * 2^-24; 2^24 / 255 is in the accumulator scale) and written to tensor
//     memory.  The two horizontal taps are stacked along N = 64; the epilogue adds its neighbour lane's upper half
//     (lane quarters overlap by one lane).
//   * conv2 and conv3 are sums over taps of row-shifted 128 x 64 products on their input grids; both grids of an
//     environment fit one tile.  Rows outside the output extent are computed from whatever lies there and dropped.
//
// conv1's and conv2's outputs are also written to global memory: hts_policy_read_activation may ask for any step's hidden
// layers and nothing else reads them.  36 KB per observation, which a thread each stores by TMA from where they lie (as
// 32-byte stores of the epilogue warps they cost 0.3 us at n = 8, 0.9 at 256, 5 at 888).
//
// Roles: warp 0 copies, warps 1 and 4 issue the MMAs of conv1 (alternate tiles), 2 and 3 those of conv2 and conv3, 5 and 6
// store the parity taps (warp 7 is idle), then eight converter warps (four per filter
// row), eight epilogue warps for conv1 and eight for conv2 and conv3 in turn (four per half of the channels).  A tile takes
// all warps of a role: what bounds small batches, and the hand-overs of large ones, is the latency of one tile.
// Tensor clocks per environment: conv1 4 tiles x 8 x 32, conv2 32 x 48, conv3 36 x 48 = 4288 (84 x 84 frames).
#include "conv_stack_tc.cuh"
#include "tc_ptx.cuh"

namespace hts {
using namespace tc;

namespace {

constexpr int kW1Bytes = 2 * 8192, kW2Bytes = 8 * 8192, kW3Bytes = 9 * 8192, kFilters = kW1Bytes + kW2Bytes + kW3Bytes;
constexpr int kTile = 124;                              // new grid positions per conv1 tile (4 quarters x 31; one more is shared)
constexpr int kIssue1 = 2;                              // threads issuing conv1's MMAs, one per operand buffer
constexpr int kConvWarp = 8, kEpi1Warp = 16, kEpi2Warp = 24, kStackThreads = 32 * 32;
constexpr int kNAcc1 = 4;                               // conv1 accumulators
constexpr uint32_t kAcc1 = 0, kOp = 256, kAcc2 = 384, kAcc3 = 448;   // tensor-memory columns

__device__ __forceinline__ void st_global_v8(void* ptr, const uint32_t (&v)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"l"(ptr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// Frame index of batch row e: e itself, or its slot in the pool.  A slot outside the pool is recorded in the status word
// and frame 0 is read instead (the heads kernel drops that row).
__device__ __forceinline__ size_t frame_of(const ConvStackParams& p, int e)
{
    if (!p.slots) return (size_t)e;
    const int sl = p.slots[e];
    if ((unsigned)sl >= (unsigned)p.pool) { atomicCAS(p.status, 0, kStatusBadSlot); return 0; }
    return (size_t)sl;
}
// 16 output channels: scale, bias, ReLU, fp16 (clamped at the largest finite value)
__device__ __forceinline__ void finish16(const uint32_t* v, float inv, const float* bias, uint32_t (&pk)[8])
{
#pragma unroll
    for (int h = 0; h < 8; ++h) {
        float x0 = __uint_as_float(v[2 * h]), x1 = __uint_as_float(v[2 * h + 1]);
        fma2(x0, x1, inv, bias[2 * h], bias[2 * h + 1]);
        pk[h] = relu_pack_h2(x0, x1);
    }
}

// WC: the frame width when known at compile time (the converter's loads then use immediate offsets), 0 = any.
// 1024 threads leave 64 registers to each: the compiler spills 8 bytes.
template <int WC>
__global__ void __launch_bounds__(kStackThreads)
conv_stack_kernel(const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2,
                  const __grid_constant__ CUtensorMap tmW3, const __grid_constant__ CUtensorMap tmT1, const __grid_constant__ CUtensorMap tmT2,
                  const ConvStackParams p)
{
    extern __shared__ uint8_t smem_raw[];
    constexpr int kStackBars = 3 + 2 + 4 + 2 * kNAcc1 + 8;
    __shared__ uint64_t bars[kStackBars];
    uint64_t *w_bar = bars, *raw_full = w_bar + 3, *raw_empty = raw_full + 1, *op_full = raw_empty + 1, *op_empty = op_full + 2,
             *acc1_full = op_empty + 2, *acc1_empty = acc1_full + kNAcc1, *a1_full = acc1_empty + kNAcc1, *a1_empty = a1_full + 1,
             *acc2_full = a1_empty + 1, *acc2_empty = acc2_full + 1, *a2_full = acc2_empty + 1, *acc3_full = a2_full + 1, *acc3_empty = acc3_full + 1, *a2_stored = acc3_empty + 1;
    __shared__ __align__(16) float s_b1[32], s_b2[64], s_b3[64];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    volatile int* abortp = &abort_flag;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t a1_addr = base + kFilters, a2_addr = a1_addr + 2 * p.a1_plane;
    uint8_t* s_raw = sm + kFilters + 2 * p.a1_plane + p.a2_bytes;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int W = WC ? WC : p.W, Ws = WC ? WC / 4 : p.Ws;
    const int envs = blockIdx.x < p.n ? (p.n - blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;   // of this CTA
    const int total = envs * p.tiles;                   // conv1 tiles of this CTA

    if (warp == 0) {
        // one barrier a lane; eight warps arrive at raw_empty, op_full, acc1_empty, a1_full, acc2_empty, a2_full and acc3_empty,
        // and at a1_empty both who reads conv1's output: the tensor core and the store
        static_assert(kStackBars == 25 && kNAcc1 == 4, "the mask");
        constexpr uint32_t eight = 1u << 4 | 3u << 5 | 15u << 13 | 1u << 17 | 1u << 20 | 1u << 21 | 1u << 23;
        if (lane < kStackBars) mbar_init(&bars[lane], eight >> lane & 1 ? 8 : lane == 18 ? 2 : 1);
        fence_barrier_init();
        __syncwarp();
        if (lane == 0) {                                 // the filters: not the previous kernel's, see `dependent`
            mbar_arrive_expect_tx(&w_bar[0], kW1Bytes);
            for (int g = 0; g < 2; ++g) tma_load_2d(sm + g * 8192, &tmW1, 0, g * 64, &w_bar[0]);
            mbar_arrive_expect_tx(&w_bar[1], kW2Bytes);
            for (int g = 0; g < 8; ++g) tma_load_2d(sm + kW1Bytes + g * 8192, &tmW2, g * 64, 0, &w_bar[1]);
            mbar_arrive_expect_tx(&w_bar[2], kW3Bytes);
            for (int g = 0; g < 9; ++g) tma_load_2d(sm + kW1Bytes + kW2Bytes + g * 8192, &tmW3, g * 64, 0, &w_bar[2]);
        }
    } else if (warp == 1) {
        tmem_alloc(&tmem_slot, 512);
    } else if (warp == 2 && lane == 0) {
        abort_flag = 0;
    }
    // positions of an odd-sized grid's border are never written: they must hold finite numbers
    for (int i = threadIdx.x; i < (2 * p.a1_plane + p.a2_bytes) / 16; i += kStackThreads) st_shared_v4(a1_addr + 16 * i, 0, 0, 0, 0);
    fence_async_proxy();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tmem_slot;
    pdl_wait();
    pdl_trigger();

    // Every barrier carries one parity bit.  A waiter is never two phases from its barrier: a frame is overwritten only
    // after all converter warps have arrived for it, conv1's output only after conv2 has read it, and the operand and
    // accumulator pairs are handed back before they are filled again.
    if (warp == 0) {
        if (lane == 0) {
            const uint32_t bytes = 4u * (uint32_t)(p.H * W);
            size_t frame = envs ? frame_of(p, blockIdx.x) : 0;
            for (int i = 0; i < envs; ++i) {
                if (!mbar_wait(raw_empty, ((uint32_t)i & 1u) ^ 1u, abortp, p.status, 41)) break;
                mbar_arrive_expect_tx(raw_full, bytes);
                bulk_load(s_raw, p.obs + frame * bytes, bytes, raw_full);
                if (i + 1 < envs) {                      // the next frame at least as far as L2
                    frame = frame_of(p, blockIdx.x + (i + 1) * gridDim.x);
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p.obs + frame * bytes), "r"(bytes) : "memory");
                }
            }
        }
    } else if (warp == 1 || warp == 4) {
        if (elect_one()) {
            constexpr uint32_t idesc = instr_desc_f16(0, 128, 64);
            const uint64_t b0 = smem_desc_sw128(base), b1 = smem_desc_sw128(base + 8192);
            bool alive = mbar_wait(&w_bar[0], 0, abortp, p.status, 42);
            for (int k = warp == 4; alive && k < total; k += kIssue1) {
                const int b = k & 1, acc = k % kNAcc1;
                if (!mbar_wait(&op_full[b], (uint32_t)(k >> 1) & 1u, abortp, p.status, 43)) break;
                if (!mbar_wait(&acc1_empty[acc], ((uint32_t)(k / kNAcc1) & 1u) ^ 1u, abortp, p.status, 44)) break;
                tc_fence_after();
                const uint32_t d = tm + kAcc1 + acc * 64, a = tm + kOp + b * 64;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) mma_f16_ts(d, a + 8 * kk, b0 + 2 * kk, idesc, kk != 0);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) mma_f16_ts(d, a + 32 + 8 * kk, b1 + 2 * kk, idesc, 1);
                mma_commit(&op_empty[b]);
                mma_commit(&acc1_full[acc]);
            }
        }
    } else if (warp == 2) {
        if (elect_one()) {
            constexpr uint32_t idesc = instr_desc_f16(0, 128, 64);
            const uint32_t w2 = base + kW1Bytes;
            bool alive = mbar_wait(&w_bar[1], 0, abortp, p.status, 42);
            for (int i = 0; alive && i < envs; ++i) {
                const uint32_t ph = (uint32_t)i & 1u;
                if (!mbar_wait(a1_full, ph, abortp, p.status, 45)) break;
                if (!mbar_wait(acc2_empty, ph ^ 1u, abortp, p.status, 46)) break;
                tc_fence_after();
#pragma unroll
                for (int tap = 0; tap < 4; ++tap) {
                    const uint32_t row = (uint32_t)((tap >> 1) * p.W1s + (tap & 1));
#pragma unroll
                    for (int pl = 0; pl < 2; ++pl) {
                        const uint64_t a = smem_desc_sw128(a1_addr + pl * p.a1_plane + row * 128), b = smem_desc_sw128(w2 + (tap * 2 + pl) * 8192);
#pragma unroll
                        for (int k = 0; k < 4; ++k) mma_f16_ss(tm + kAcc2, a + 2 * k, b + 2 * k, idesc, (tap | pl | k) != 0);
                    }
                }
                mma_commit(a1_empty);
                mma_commit(acc2_full);
            }
        }
    } else if (warp == 3) {
        if (elect_one()) {
            constexpr uint32_t idesc = instr_desc_f16(0, 128, 64);
            const uint32_t w3 = base + kW1Bytes + kW2Bytes;
            bool alive = mbar_wait(&w_bar[2], 0, abortp, p.status, 42);
            for (int i = 0; alive && i < envs; ++i) {
                const uint32_t ph = (uint32_t)i & 1u;
                if (!mbar_wait(a2_full, ph, abortp, p.status, 47)) break;
                if (!mbar_wait(acc3_empty, ph ^ 1u, abortp, p.status, 48)) break;
                tc_fence_after();
#pragma unroll
                for (int tap = 0; tap < 9; ++tap) {
                    const uint32_t row = (uint32_t)((tap / 3) * p.W2 + tap % 3);
                    const uint64_t a = smem_desc_sw128(a2_addr + row * 128), b = smem_desc_sw128(w3 + tap * 8192);
#pragma unroll
                    for (int k = 0; k < 4; ++k) mma_f16_ss(tm + kAcc3, a + 2 * k, b + 2 * k, idesc, (tap | k) != 0);
                }
                mma_commit(acc3_full);                  // also says that conv2's output has been read: it is written after this wait
            }
        }
    } else if (warp == 5 || warp == 6) {
        // ---- parity taps: the SM's copy of a layer, as it lies there
        if (lane == 0) {
            for (int i = 0; i < envs; ++i) {
                const int e = p.row0 + (int)(blockIdx.x + i * gridDim.x);
                if (!mbar_wait(warp == 5 ? a1_full : a2_full, (uint32_t)i & 1u, abortp, p.status, 57)) break;
                if (warp == 5) {
                    for (int pl = 0; pl < 2; ++pl) tma_store_4d(&tmT1, a1_addr + pl * p.a1_plane, pl * 64, 0, e, 0);
                } else {
                    tma_store_4d(&tmT2, a2_addr, 0, 0, e, 0);
                }
                tma_store_commit();
                tma_store_wait_read();
                mbar_arrive(warp == 5 ? a1_empty : a2_stored);
            }
            tma_store_wait();
        }
    } else if (warp >= kConvWarp && warp < kEpi1Warp) {
        // ---- converters: warps of group dy write the operand of that filter row
        const int dy = (warp - kConvWarp) >> 2, qq = warp & 3;
        const int cells = Ws * (p.H / 4);
        for (int k = 0, t = 0, i = 0; k < total; ++k) {
            const int b = k & 1;
            int q = t * kTile + 31 * qq + lane + dy * Ws;
            q = q < cells ? q : 0;                       // past the last position: results are never stored
            const int Y = q / Ws, X = q - Y * Ws;
            const uint8_t* src = s_raw + (4 * Y) * W + 4 * X;
            if (t == 0 && !mbar_wait_warp(raw_full, (uint32_t)i & 1u, abortp, p.status, 51)) break;
            uint32_t v[32];
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int uy = 0; uy < 4; ++uy) {
                    const uint32_t w = *reinterpret_cast<const uint32_t*>(src + (c * p.H + uy) * W);
                    v[c * 8 + uy * 2] = __byte_perm(w, 0u, 0x4140);
                    v[c * 8 + uy * 2 + 1] = __byte_perm(w, 0u, 0x4342);
                }
            if (++t == p.tiles) {                        // this warp has read the frame for the last time
                t = 0;
                ++i;
                __syncwarp();
                if (lane == 0) mbar_arrive(raw_empty);
            }
            if (!mbar_wait_warp(&op_empty[b], ((uint32_t)(k >> 1) & 1u) ^ 1u, abortp, p.status, 52)) break;
            tc_fence_after();
            tmem_st_32x32(tm + kOp + b * 64 + dy * 32 + ((uint32_t)(qq * 32) << 16), v);
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&op_full[b]);
        }
    } else if (warp >= kEpi1Warp && warp < kEpi2Warp) {
        // ---- conv1 epilogue: warps of group h take output channels [16 h, 16 h + 16)
        const int h = (warp - kEpi1Warp) >> 2, qq = warp & 3;
        const float inv = *p.inv1;
        s_b1[lane] = p.b1[lane];                         // every warp of the role writes the same
        __syncwarp();
        const uint32_t lanes = ((uint32_t)(qq * 32) << 16) + 16 * h;
        for (int k = 0, t = 0, i = 0; k < total; ++k) {
            const int q = t * kTile + 31 * qq + lane, y = q / Ws, x = q - y * Ws, acc = k % kNAcc1;
            const bool valid = lane < 31 && y < p.H1 && x < p.W1;
            const int row = (y >> 1) * p.W1s + (x >> 1);
            const uint32_t dst = a1_addr + (y & 1) * p.a1_plane + row * 128, swz = (uint32_t)(row & 7), ch = (uint32_t)((x & 1) * 4 + 2 * h);
            const uint32_t taddr = tm + kAcc1 + acc * 64 + lanes;
            if (!mbar_wait_warp(&acc1_full[acc], (uint32_t)(k / kNAcc1) & 1u, abortp, p.status, 53)) break;
            tc_fence_after();
            uint32_t v0[16], v1[16], pk[8];
            tmem_ld_32x16(taddr, v0);                    // dx = 0 part of this position's output
            tmem_ld_32x16(taddr + 32, v1);               // dx = 1 part of the output one position to the left
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc1_empty[acc]);
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
                float a0 = __uint_as_float(v0[c]), a1 = __uint_as_float(v0[c + 1]);
                add2(a0, a1, __shfl_down_sync(0xffffffffu, __uint_as_float(v1[c]), 1), __shfl_down_sync(0xffffffffu, __uint_as_float(v1[c + 1]), 1));
                v0[c] = __float_as_uint(a0); v0[c + 1] = __float_as_uint(a1);
            }
            finish16(v0, inv, s_b1 + 16 * h, pk);
            // finished in registers: conv2 and the store have until here to read the previous environment's rows
            if (t == 0 && i > 0 && !mbar_wait_warp(a1_empty, (uint32_t)(i - 1) & 1u, abortp, p.status, 54)) break;
            if (valid) {
                st_shared_v4(dst + ((ch ^ swz) << 4), pk[0], pk[1], pk[2], pk[3]);
                st_shared_v4(dst + (((ch + 1) ^ swz) << 4), pk[4], pk[5], pk[6], pk[7]);
            }
            if (++t == p.tiles) {
                t = 0;
                ++i;
                fence_async_proxy();                     // the tensor core reads these rows through the asynchronous proxy
                __syncwarp();
                if (lane == 0) mbar_arrive(a1_full);
            }
        }
    } else if (warp >= kEpi2Warp) {
        // ---- conv2 and conv3 epilogues: thread = row of the input grid, warps of group h take channels [32 h, 32 h + 32)
        const int h = (warp - kEpi2Warp) >> 2, qq = warp & 3, m = qq * 32 + lane;
        const float inv2 = *p.inv2, inv3 = *p.inv3;
        for (int i = lane; i < 64; i += 32) { s_b2[i] = p.b2[i]; s_b3[i] = p.b3[i]; }      // every warp of the role writes the same
        __syncwarp();
        const uint32_t lanes = ((uint32_t)(qq * 32) << 16) + 32 * h;
        const int y2 = m / p.W1s, x2 = m - y2 * p.W1s, y3 = m / p.W2, x3 = m - y3 * p.W2;
        const bool ok2 = y2 < p.H2 && x2 < p.W2, ok3 = y3 < p.H3 && x3 < p.W3;
        const int r2 = y2 * p.W2 + x2;
        const uint32_t dst2 = a2_addr + r2 * 128, swz = (uint32_t)(r2 & 7);
        for (int i = 0; i < envs; ++i) {
            const uint32_t ph = (uint32_t)i & 1u;
            const size_t e = (size_t)p.row0 + blockIdx.x + (size_t)i * gridDim.x;
            uint32_t v[32], pk[2][8];
            if (!mbar_wait_warp(acc2_full, ph, abortp, p.status, 55)) break;
            tc_fence_after();
            tmem_ld_32x32(tm + kAcc2 + lanes, v);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc2_empty);
            if (i > 0 && !mbar_wait_warp(a2_stored, (uint32_t)(i - 1) & 1u, abortp, p.status, 58)) break;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                finish16(v + 16 * j, inv2, s_b2 + 32 * h + 16 * j, pk[j]);
                if (ok2) {
                    const uint32_t ch = (uint32_t)(4 * h + 2 * j);
                    st_shared_v4(dst2 + ((ch ^ swz) << 4), pk[j][0], pk[j][1], pk[j][2], pk[j][3]);
                    st_shared_v4(dst2 + (((ch + 1) ^ swz) << 4), pk[j][4], pk[j][5], pk[j][6], pk[j][7]);
                }
            }
            fence_async_proxy();
            __syncwarp();
            if (lane == 0) mbar_arrive(a2_full);
            if (!mbar_wait_warp(acc3_full, ph, abortp, p.status, 56)) break;
            tc_fence_after();
            tmem_ld_32x32(tm + kAcc3 + lanes, v);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc3_empty);
            __half* out = p.a3 + (e * p.P3 + (size_t)(y3 * p.W3 + x3)) * 64 + 32 * h;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                finish16(v + 16 * j, inv3, s_b3 + 32 * h + 16 * j, pk[0]);
                if (ok3) st_global_v8(out + 16 * j, pk[0]);
            }
        }
    }
    if (*abortp) {                                       // give copies still in flight time to land
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tm, 512);
}

template <int WC>
hts_status launch(const CUtensorMap& w1, const CUtensorMap& w2, const CUtensorMap& w3, const CUtensorMap& t1, const CUtensorMap& t2, const ConvStackParams& p, int smem, int grid,
                  bool dependent, cudaStream_t s)
{
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(conv_stack_kernel<WC>, allowed));
    HTS_CUDA(launch_chained(dependent, conv_stack_kernel<WC>, dim3(grid), dim3(kStackThreads), (size_t)smem, s, w1, w2, w3, t1, t2, p));
    note_launch();
    return HTS_OK;
}

inline int stack_smem(const ConvStackParams& p) { return 1024 + kFilters + 2 * p.a1_plane + p.a2_bytes + p.raw_bytes; }

}  // namespace

bool conv_stack_plan(const Geometry& g, ConvStackParams* p)
{
    if (g.C != 4 || g.H % 4 || g.W % 4) return false;
    p->H = g.H; p->W = g.W; p->Ws = g.W / 4;
    p->H1 = g.H1; p->W1 = g.W1; p->W1s = (g.W1 + 1) / 2; p->P1s = p->W1s * ((g.H1 + 1) / 2);
    p->H2 = g.H2; p->W2 = g.W2; p->P2 = g.H2 * g.W2; p->H3 = g.H3; p->W3 = g.W3; p->P3 = g.H3 * g.W3;
    if ((g.H2 - 1) * p->W1s + g.W2 > 128 || (g.H3 - 1) * g.W2 + g.W3 > 128) return false;
    const int last = (g.H1 - 1) * p->Ws + g.W1;          // positions up to the last output
    p->tiles = (last + kTile - 1) / kTile;
    p->a1_plane = (p->P1s * 128 + 1023) / 1024 * 1024;
    p->a2_bytes = (p->P2 * 128 + 1023) / 1024 * 1024;
    p->raw_bytes = (4 * g.H * g.W + 1023) / 1024 * 1024;
    // the shifted tiles of conv2 and conv3 reach past their grids: into what follows, never past the allocation
    const int reach1 = p->a1_plane + (128 + p->W1s + 1) * 128, reach2 = (128 + 2 * g.W2 + 2) * 128;
    if (reach1 > 2 * p->a1_plane + p->a2_bytes + p->raw_bytes || reach2 > p->a2_bytes + p->raw_bytes) return false;
    return stack_smem(*p) <= 226 * 1024;
}

hts_status conv_stack_launch(const CUtensorMap& w1, const CUtensorMap& w2, const CUtensorMap& w3, const CUtensorMap& t1, const CUtensorMap& t2,
                             const ConvStackParams& p, bool dependent, cudaStream_t s)
{
    const int sms = device_sm_count(device_slot()), grid = p.n < sms ? p.n : sms, smem = stack_smem(p);
    return p.W == 84 ? launch<84>(w1, w2, w3, t1, t2, p, smem, grid, dependent, s) : launch<0>(w1, w2, w3, t1, t2, p, smem, grid, dependent, s);
}

}  // namespace hts
