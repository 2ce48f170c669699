// conv2 / conv3 of the policy-value network as a persistent tcgen05 kernel.
//
// Activations are rows of 64 channels (128 bytes) in the order (y, environment, x).  An M tile is 128 consecutive columns
// (environment, x) of the batch, and the kernel marches down the grid rows: input row y of a tile is loaded once (one TMA box
// per 64-channel plane, 128-byte swizzle, KX - 1 columns wider) and contributes to the KY output rows y - KY + 1 .. y.  The
// filter sits in shared memory with the vertical taps stacked along N, so ONE instruction multiplies the input row by KY taps
// into KY accumulators that lie side by side in tensor memory; the horizontal taps read the same tile through a descriptor
// moved by dx rows (128 bytes each; the swizzle follows the address bits).
//
// Why: a 128 x 64 x 16 instruction with both operands in shared memory takes 48 clocks (128 + 64 operand rows of 32 bytes at
// 128 bytes a clock) where its products need 32; with N = 128 fetch and products take 64 clocks each, with N = 192 the
// products' 96 exceed the fetch.  And no grid row is multiplied that no output needs (conv3: 7 of 9 columns are outputs instead
// of 49 of 81 grid points).  A sum still runs over (dy, dx, plane, channel) in that order: the bits are those of one tap
// after the other.  Against one instruction per tap on flat tiles: step of 1024 observations 51.9 -> 48.1 us, of 1733 76.9 ->
// 71.5, of 8192 243 -> 224 (conv3 46 -> 29; conv2 52 -> 49, where 210 MB of input and 85 of output at 6 TB/s are the bound), of
// 512 football frames 51.6 -> 51.1.  conv2's instructions take 80 clocks instead of 64 while copies write the same shared memory.
//
// Work: output rows of all tiles in a line, cut into one stretch per CTA; a stretch enters each tile it touches with KY - 1
// rows more than it puts out.  Eight accumulators of 64 columns form a ring over the CTA's output rows; a group of rows that
// crosses the ring's end takes two instructions.  One thread issues all MMAs (two would have to order their sums), four
// groups of four warps drain accumulators c, c + 4.
#include "conv_res_tc.cuh"
#include "tc_ptx.cuh"

namespace hts {
using namespace tc;

namespace {

constexpr int kRing = 8;                        // accumulators in tensor memory (64 columns each)
constexpr int kGroups = 4;                      // epilogue groups of four warps
constexpr int kThreads = 128 + kGroups * 128;   // warp 0 copies, warp 1 issues MMAs, warps 2 and 3 idle, then the epilogues
constexpr int kPlaneBytes = 17 * 1024;          // one plane of an input row: at most 136 rows of 128 bytes

template <int KY, int KX, int CPT> struct RowsShape {
    static constexpr int kFilter = KY * KX * CPT * 64 * 128;
    static constexpr int kStage = CPT * kPlaneBytes;
    static constexpr int kStages = (226 * 1024 - kFilter) / kStage;
    static constexpr int kSmem = 1024 + kFilter + kStages * kStage;
    static_assert(kConvRowsBox<KX> * 128 <= kPlaneBytes && kStages >= 2, "an input row does not fit its stage");
};

// 256-bit store of eight packed half2 (one 32-byte sector)
__device__ __forceinline__ void st_global_v8(void* ptr, const uint32_t (&v)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"l"(ptr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}

template <int KY, int KX, int CPT>
__global__ void __launch_bounds__(kThreads)
conv_rows_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const ConvRowsParams p)
{
    using S = RowsShape<KY, KX, CPT>;
    constexpr int NST = S::kStages;
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bars[1 + 2 * NST + 2 * kRing];
    uint64_t *w_bar = bars, *a_full = bars + 1, *a_empty = a_full + NST, *d_full = a_empty + NST, *d_empty = d_full + kRing;
    __shared__ float s_bias[64];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    volatile int* abortp = &abort_flag;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this CTA's stretch of output rows (tile, y)
    const int H = p.H_out, share = p.tiles * H / (int)gridDim.x, extra = p.tiles * H - share * (int)gridDim.x;
    const int r0 = (int)blockIdx.x * share + min((int)blockIdx.x, extra), total = share + ((int)blockIdx.x < extra);
    const int tile0 = r0 / H, y0 = r0 - tile0 * H;

    // The prologue is on the step's critical path: this CTA gets the SM when the previous kernel's last one leaves it.
    if (warp == 0) {
        for (int i = lane; i < 1 + 2 * NST + 2 * kRing; i += 32) mbar_init(&bars[i], i < 1 + 2 * NST + kRing ? 1 : 4);
        fence_barrier_init();
        __syncwarp();
        if (lane == 0) {                                 // the filter does not depend on the previous kernel
            mbar_arrive_expect_tx(w_bar, S::kFilter);
            for (int dx = 0; dx < KX; ++dx)
                for (int pl = 0; pl < CPT; ++pl)
                    for (int dy = 0; dy < KY; ++dy)      // the last filter row first: it belongs to the earliest output row
                        tma_load_2d(sm + ((dx * CPT + pl) * KY + KY - 1 - dy) * 8192, &tmW, ((dy * KX + dx) * CPT + pl) * 64, 0, w_bar);
        }
    } else if (warp == 1) {
        tmem_alloc(&tmem_slot, kRing * 64);
    } else if (warp == 2 && lane == 0) {
        abort_flag = 0;
        tma_prefetch_desc(&tmA);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_d = tmem_slot;
    pdl_wait();
    pdl_trigger();

    if (warp == 0) {
        if (lane == 0) {
            int st = 0, tile = tile0, y = y0;            // input row y of the tile
            uint32_t ph = 1;
            for (int left = total; left > 0;) {
                const int cnt = min(left, H - y);        // output rows in this tile
                int row = y * p.in_plane + p.col0 + tile * 128;
                for (int i = 0; i < cnt + KY - 1; ++i, row += p.in_plane) {
                    if (!mbar_wait(&a_empty[st], ph, abortp, p.status, 21)) { left = 0; break; }
                    uint8_t* dst = sm + S::kFilter + st * S::kStage;
                    mbar_arrive_expect_tx(&a_full[st], (uint32_t)(CPT * kConvRowsBox<KX> * 128));
                    for (int pl = 0; pl < CPT; ++pl) tma_load_2d(dst + pl * kPlaneBytes, &tmA, pl * 64, row, &a_full[st]);
                    if (++st == NST) { st = 0; ph ^= 1u; }
                }
                left -= cnt;
                ++tile;
                y = 0;
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            constexpr uint32_t idesc0 = instr_desc_f16(0, 128, 0);
            constexpr int KS = KX * CPT * 4;             // K steps of an input row: (dx, plane, 16 channels)
            // an input row: stage and its phase; its place i in the tile's stretch of cnt output rows, c0 of them before
            int st = 0, i = 0, c0 = 0, cnt = min(total, H - y0);
            uint32_t ph = 0;
            auto start_wait = [&](bool a_there, bool d_there) {
                if (!a_there && !mbar_wait(&a_full[st], ph, abortp, p.status, 23)) return false;
                const int cy = c0 + i;
                return d_there || i >= cnt || mbar_wait(&d_empty[cy % kRing], (((uint32_t)(cy / kRing)) & 1u) ^ 1u, abortp, p.status, 24);
            };
            bool alive = mbar_wait(w_bar, 0, abortp, p.status, 22) && start_wait(false, false);
            while (alive) {                              // input row i feeds outputs i - KY + 1 .. i
                const int lo = i - KY + 1 > 0 ? i - KY + 1 : 0, hi = i < cnt ? i : cnt - 1, m = hi - lo + 1;
                const int slot = (c0 + lo) % kRing;
                const int m1 = m < kRing - slot ? m : kRing - slot, m2 = m - m1;   // accumulators up to the ring's end, and past it
                const uint64_t a = smem_desc_sw128(base + S::kFilter + st * S::kStage);
                const uint64_t b = smem_desc_sw128(base + (KY - 1 - (i - lo)) * 8192);
                const uint32_t d = tmem_d + slot * 64;
                auto issue = [&](int kk, uint32_t dd, int skip, int count, uint32_t acc) {
                    const int g = kk >> 2;
                    mma_f16_ss(dd, a + (uint32_t)((g % CPT) * (kPlaneBytes >> 4) + (g / CPT) * 8 + 2 * (kk & 3)),
                               b + (uint32_t)(g * KY * 512 + 2 * (kk & 3)) + (uint64_t)(skip * 512), idesc0 + ((uint32_t)count << 20), acc);
                };
                tc_fence_after();
                if (i < cnt) {                           // output row i starts here: its accumulator takes its first product by itself
                    const int o1 = m - 1 < m1 ? m - 1 : m1;
                    if (o1 > 0) issue(0, d, 0, o1, 1);
                    if (m - 1 > o1) issue(0, tmem_d, o1, m - 1 - o1, 1);
                    issue(0, tmem_d + ((c0 + i) % kRing) * 64, m - 1, 1, 0);
                } else {
                    issue(0, d, 0, m1, 1);
                    if (m2 > 0) issue(0, tmem_d, m1, m2, 1);
                }
                if (m2 > 0) {
#pragma unroll 1                                    // seldom taken: unrolled, its code cost a small batch 0.3 us
                    for (int kk = 1; kk < KS; ++kk) issue(kk, tmem_d, m1, m2, 1);
                }
#pragma unroll
                for (int kk = 1; kk < KS / 2; ++kk) issue(kk, d, 0, m1, 1);
                // The next row's barriers are polled while this row's instructions execute: the tensor core takes about four
                // ahead, and a poll lasts over 100 clocks in the shared memory that it fetches its operands from.
                const int stage = st, done = i - KY + 1 >= 0 ? (c0 + i - KY + 1) % kRing : -1;
                if (++st == NST) { st = 0; ph ^= 1u; }
                if (++i == cnt + KY - 1) { c0 += cnt; i = 0; cnt = min(total - c0, H); }
                const bool more = c0 < total;
                bool a_there = false, d_there = false;
                if (more) {
                    a_there = mbar_test(&a_full[st], ph);
                    const int cy = c0 + i;
                    if (i < cnt) d_there = mbar_test(&d_empty[cy % kRing], (((uint32_t)(cy / kRing)) & 1u) ^ 1u);
                }
#pragma unroll
                for (int kk = KS / 2; kk < KS; ++kk) issue(kk, d, 0, m1, 1);
                mma_commit(&a_empty[stage]);
                if (done >= 0) mma_commit(&d_full[done]);
                alive = more && start_wait(a_there, d_there);
            }
        }
    } else if (warp >= 4) {
        const int grp = (warp - 4) >> 2;
        const int q = warp & 3;                         // TMEM lane quarter this warp may read
        const float inv = *p.inv_scale;
        s_bias[lane] = p.bias[lane];                    // every epilogue warp writes the same
        s_bias[32 + lane] = p.bias[32 + lane];
        __syncwarp();
        int tile = tile0, y = y0 + grp, at = -1;
        bool valid = false;
        __half* dst = nullptr;
        for (int c = grp; c < total; c += kGroups, y += kGroups) {
            while (y >= H) { y -= H; ++tile; }
            if (at != tile) {                           // this thread's column of the new tile
                at = tile;
                const int col = tile * 128 + q * 32 + lane, env = col / p.W_in, x = col - env * p.W_in;
                valid = env < p.n_env && x < p.W_out;
                dst = p.out + (size_t)env * p.out_env + (size_t)x * 64;
            }
            const int slot = c % kRing;
            if (!mbar_wait_warp(&d_full[slot], ((uint32_t)(c / kRing)) & 1u, abortp, p.status, 25)) break;
            tc_fence_after();
            uint32_t v0[32], v1[32];
            const uint32_t taddr = tmem_d + slot * 64 + ((uint32_t)(q * 32) << 16);
            tmem_ld_32x32(taddr, v0);
            tmem_ld_32x32(taddr + 32, v1);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&d_empty[slot]);  // accumulator is in registers: hand it back
            if (valid) {
                __half* o = dst + (size_t)y * p.out_y;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
#pragma unroll
                    for (int j = 0; j < 32; j += 16) {
                        uint32_t pk[8];
#pragma unroll
                        for (int h = 0; h < 8; ++h) {
                            const int k = j + 2 * h;
                            float x0 = __uint_as_float(half ? v1[k] : v0[k]);
                            float x1 = __uint_as_float(half ? v1[k + 1] : v0[k + 1]);
                            fma2(x0, x1, inv, s_bias[half * 32 + k], s_bias[half * 32 + k + 1]);
                            pk[h] = relu_pack_h2(x0, x1);     // ReLU, round to fp16, clamp at the largest finite value
                        }
                        st_global_v8(o + half * 32 + j, pk);
                    }
                }
            }
        }
    }
    if (*abortp) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_d, kRing * 64);
}

}  // namespace

template <int KY, int KX, int CPT>
hts_status conv_rows_launch(const CUtensorMap& act_map, const CUtensorMap& weight_map, const ConvRowsParams& p, cudaStream_t s)
{
    using S = RowsShape<KY, KX, CPT>;
    const int sm_count = device_sm_count(device_slot());
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(conv_rows_kernel<KY, KX, CPT>, allowed));
    const int rows = p.tiles * p.H_out, grid = rows < sm_count ? rows : sm_count;
    HTS_CUDA(launch_pdl(conv_rows_kernel<KY, KX, CPT>, dim3(grid), dim3(kThreads), (size_t)S::kSmem, s, act_map, weight_map, p));
    note_launch();
    return HTS_OK;
}

template hts_status conv_rows_launch<2, 2, 2>(const CUtensorMap&, const CUtensorMap&, const ConvRowsParams&, cudaStream_t);
template hts_status conv_rows_launch<3, 3, 1>(const CUtensorMap&, const CUtensorMap&, const ConvRowsParams&, cudaStream_t);

}  // namespace hts
