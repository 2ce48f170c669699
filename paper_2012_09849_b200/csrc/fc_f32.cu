// fp32 dense layer of the actor step for batches that fill the device.
//
// Lane l of a warp runs chain l of TE rows x TO outputs, so both operands are contiguous across the lanes; one transposing
// reduction closes the tree (at each level a lane keeps half of its values and gets its partner's share of them).  Stages of 256
// columns arrive as boxes of 16 rows x 128, asked for by a warp of their own (all waits are bounded).  A stage's eight steps are one
// straight run of instructions, so that a step's loads are under way during the products before it; what remains is the first
// step of each stage, and loads from shared memory, a clock for each of the 16 words that 64 multiply-adds take, beside as much time
// in the fp32 pipes.  Whole fp32 step of 84 x 84 x 4, us at 40 / 80 / 160 / 256 / 512 / 1024 rows: 42.3 / 60.3 / 91.3 / 124 / 216 / 406; with
// stages of 128 columns and the next step's loads written out before a step's products 45.3 / 62.6 / 94.3 / 129 / 223 / 421 (straight
// runs of 128: 44.6 / 62.3 / 93.6 / 128 / 221 / 417; the next stage's first loads before a stage's last products: 44.2 / 61.0 / 92.5 /
// 126 / 218 / 412; 8 x 4 per warp and eight warps: 43.3 / 62.0 / 95.3 / 129 / 225 / 426; 16 x 8, two warps per scheduler: 52 / 66 / 101 /
// 128 / 230 / 423).  A copy per row instead of a box: 70 clocks each.
#include "common.cuh"
#include "f32x2.cuh"
#include "fc_f32.cuh"
#include "tc_host.cuh"
#include "tc_ptx.cuh"

namespace hts {
namespace {

template <int TE, int TO, int WE, int WO, int SUB, int NST, int PER_SM>
__global__ void __launch_bounds__(32 * (WE * WO + 1), PER_SM)
fc_lanes_kernel(const FcParams p, const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mw)
{
    constexpr int COLS = kFcBoxCols, BOX = kFcBoxRows, NC = WE * WO, RX = TE * WE, RW = TO * WO, BOXES = (RX + RW) * COLS, STAGE = SUB * BOXES, NV = TE * TO;
    static_assert(RX % BOX == 0 && RW % BOX == 0, "whole boxes");
    extern __shared__ float s_dyn[];
    float* s_ring = s_dyn + (-tc::smem_u32(s_dyn) & 127) / 4;                    // [NST][SUB][RX + RW][COLS]
    __shared__ uint64_t full[NST], freed[NST];
    __shared__ int abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < NST; ++i) { tc::mbar_init(full + i, 1); tc::mbar_init(freed + i, NC); }
        abort_flag = 0;
        tc::fence_barrier_init();
    }
    __syncthreads();
    const int stages = (p.F + SUB * COLS - 1) / (SUB * COLS), e_base = blockIdx.y * RX, o_base = blockIdx.x * RW;
    if (warp == NC) {
        pdl_wait();
        int st = 0;
#pragma unroll 1
        for (; st < stages; ++st) {
            const int slot = st % NST;
            if (st >= NST && !tc::mbar_wait_warp(freed + slot, (st / NST - 1) & 1, &abort_flag, p.status, 50)) break;
            if (lane == 0) tc::mbar_arrive_expect_tx(full + slot, STAGE * 4);
            __syncwarp();
            if (lane < SUB * (RX + RW) / BOX) {         // columns past the last are zeros
                const int r = lane / SUB * BOX, sub = lane % SUB, c = (st * SUB + sub) * COLS;
                float* dst = s_ring + slot * STAGE + sub * BOXES + r * COLS;
                if (r < RX) tc::tma_load_2d(dst, &mx, c, p.row0 + e_base + r, full + slot);
                else tc::tma_load_2d(dst, &mw, c, o_base + r - RX, full + slot);
            }
        }
        if (st < stages) tc::let_copies_land();
        return;
    }
    const int we = warp % WE, wo = warp / WE;
    f32x2 acc[TE / 2][TO];
#pragma unroll
    for (int i = 0; i < TE / 2; ++i)
#pragma unroll
        for (int j = 0; j < TO; ++j) acc[i][j] = 0;
    pdl_wait();                                          // here, so that the waits' limit does not count the kernel before
#pragma unroll 1
    for (int st = 0; st < stages; ++st) {
        const int slot = st % NST;
        if (!tc::mbar_wait_warp(full + slot, (st / NST) & 1, &abort_flag, p.status, 52)) {
            tc::let_copies_land();
            break;
        }
        const float* xr = s_ring + slot * STAGE + we * TE * COLS + lane;
        const float* wr = s_ring + slot * STAGE + (RX + wo * TO) * COLS + lane;
        auto step = [&](int c) {
            f32x2 xx[TE / 2];
            float wv[TO];
#pragma unroll
            for (int j = 0; j < TO; ++j) wv[j] = wr[j * COLS + c];
#pragma unroll
            for (int i = 0; i < TE / 2; ++i) xx[i] = pair(xr[2 * i * COLS + c], xr[(2 * i + 1) * COLS + c]);
#pragma unroll
            for (int j = 0; j < TO; ++j) {
                const f32x2 ww = both(wv[j]);
#pragma unroll
                for (int a = 0; a < TE / 2; ++a) {
                    const int i = j & 1 ? TE / 2 - 1 - a : a;
                    fma2(acc[i][j], xx[i], ww);
                }
            }
        };
        const int cols = p.F - st * SUB * COLS;          // a multiple of 64
        if (cols >= SUB * COLS) {
#pragma unroll
            for (int c = 0; c < SUB * COLS; c += 32) step(c / COLS * BOXES + c % COLS);
        } else
#pragma unroll 1
            for (int c = 0; c < cols; c += 32) step(c / COLS * BOXES + c % COLS);
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(freed + slot);
    }
    float v[NV];
#pragma unroll
    for (int i = 0; i < TE; ++i)
#pragma unroll
        for (int j = 0; j < TO; ++j) v[i * TO + j] = lane_of(acc[i / 2][j], i & 1);
    int id = 0;                                          // (row, output) of v[0]
#pragma unroll
    for (int m = 16, len = NV / 2; m > 0; m >>= 1, len >>= 1) {
        const bool up = lane & m;
#pragma unroll
        for (int k = 0; k < len; ++k) {
            const float send = up ? v[k] : v[k + len], keep = up ? v[k + len] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, m);
        }
        id += up ? len : 0;
    }
    constexpr int LEFT = NV / 32;
    static_assert(LEFT >= 1 && TO % LEFT == 0, "a lane's results are of one row");
    const int e = e_base + we * TE + id / TO, o = o_base + wo * TO + id % TO;
    if (e < p.n)
#pragma unroll
        for (int k = 0; k < LEFT; ++k) {
            const float r = v[k] + p.b[o + k];
            p.h[(size_t)e * 512 + o + k] = r > 0.f ? r : 0.f;
        }
}

template <int TE, int TO, int WE, int WO, int SUB, int NST, int PER_SM>
hts_status launch_lanes(const FcParams& p, const FcMaps& m, cudaStream_t s)
{
    constexpr int smem = NST * SUB * (TE * WE + TO * WO) * kFcBoxCols * 4 + 128;
    static_assert(smem <= 227 * 1024 / PER_SM - 1024 - 128, "shared memory");
    auto kernel = fc_lanes_kernel<TE, TO, WE, WO, SUB, NST, PER_SM>;
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(kernel, allowed));
    HTS_CUDA(launch_pdl(kernel, dim3(512 / (TO * WO), (unsigned)((p.n + TE * WE - 1) / (TE * WE))), dim3(32 * (WE * WO + 1)), (size_t)smem, s, p, m.x, m.w));
    note_launch();
    return HTS_OK;
}

}  // namespace

bool make_fc_maps(const float* x, const float* w, int F, size_t frames, FcMaps* m)
{
    m->ok = F >= kFcBoxCols;
    return !m->ok || (tc::make_f32_map(&m->x, x, frames, F, kFcBoxRows, kFcBoxCols) && tc::make_f32_map(&m->w, w, 512, F, kFcBoxRows, kFcBoxCols));
}

hts_status launch_fc_lanes(const FcParams& p, const FcMaps& m, cudaStream_t s)
{
    return m.ok ? launch_lanes<8, 8, 2, 2, 2, 2, 3>(p, m, s) : HTS_ERR_UNSUPPORTED;
}

}  // namespace hts
