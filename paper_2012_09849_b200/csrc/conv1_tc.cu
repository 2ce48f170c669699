// conv1 (8x8 / 4, C -> 32) of the policy-value network, fused from raw frames to fp16 output.
//
// An 8x8 stride-4 convolution is a 2x2 stride-1 convolution on the space-to-depth(4) image: grid
// pixel (Y, X) carries the 16 C bytes x[c][4Y+uy][4X+ux], and output pixel (y, x) is the sum over the
// four taps (dy, dx) of  pix(y+dy, x+dx) . w[o][dy][dx].  The kernel never builds im2col rows:
//
//   * The 128 rows of an MMA tile are 128 consecutive grid COLUMNS of the batch (flat index
//     q = env * Ws + X), and the kernel marches down the grid rows Y.  Grid row Y of those columns is
//     converted to fp16 once (a zero-extended byte is the fp16 subnormal b * 2^-24, exact; 2^24 / 255
//     goes into the accumulator scale), written to tensor memory and multiplied at once by all four taps:
//     as the dy = 1 row of output row Y - 1 and as the dy = 0 row of output row Y, whose accumulators lie side by side
//     (tcgen05.mma with A from tensor memory, 128 x 64 x 16 or both at once as 128 x 128 x 16).
//   * The two horizontal taps are stacked along N: accumulator columns [0, 32) hold the dx = 0 part of
//     output (y, X), columns [32, 64) the dx = 1 part, which belongs to output (y, X - 1).  The
//     epilogue adds its neighbour lane's upper half to its own lower half, applies scale, bias and
//     ReLU and stores fp16 in the layout conv2 reads.  Warp quarters overlap by one lane (quarter k
//     starts at column 31 k of the tile), so the neighbour is always in the same warp.
//
// Work: output rows of all tiles (124 new grid columns each) in a line, cut into one stretch per CTA and that into one per
// PIPE; a stretch enters each tile it touches with one grid row more than it puts out.  Where a CTA has several tiles of four
// channels, the pipes take half of each tile's rows instead: a frame on a tile's border is then still in L2 when the next tile
// needs it (convolution of 8192 frames 92 -> 85 us, of 4096 51 -> 50; with fewer rows the extra one costs more: 2048 31.2 -> 31.6).
// The pipes run side by side, each with half of tensor memory and its own barriers: what a pipe hands from role to role is an ENTRY of 128 K values per column
// (two grid rows of four channels, one of eight, or half of one of sixteen), and every hand-over, copy and loop turn costs a
// thread more than the tensor core needs for the entry, so the pipes fill each other's gaps.  In each pipe two warps stage
// entries in shared memory, four (thread = grid column) expand them into tensor memory, one thread issues their MMAs, and two
// groups of four drain alternate output rows.  All waits are bounded.
//
// Staging: one TMA box per environment (all of the entry's rows; the frames are viewed as 32-bit words so that a box row is
// the 4 W contiguous bytes under one grid row).  A thread gets a copy under way every 120 clocks at best, 250 among the other
// warps' work, whatever its size (336 bytes or 6.7 KB): one thread with six or seven boxes per tile bounded this kernel.
// Asynchronous copies by threads and loads straight into the converters' registers are slower: the L1 keeps too
// few lines in flight beside so much shared memory.
//
// Against one pipeline per CTA staged by one thread: convolution of 1024 frames of 84 x 84 19 -> 17 us, of 8192 89 -> 81 (441 MB of
// frames and output: 5.4 TB/s), of 512 football frames 29 -> 19.5, of 4096 141 -> 113 (566 MB: 5.0 TB/s).
#include "conv1_tc.cuh"
#include "tc_ptx.cuh"
#include "tc_host.cuh"

namespace hts {
using namespace tc;

namespace {

constexpr int kPipes = 2;
constexpr int kLoadWarps = 2, kEpiGroups = 2;   // per pipe: staging warps, groups of four epilogue warps
constexpr int kIssueWarp0 = kPipes * kLoadWarps, kConvWarp0 = 8, kEpiWarp0 = kConvWarp0 + 4 * kPipes;
constexpr int kThreads = (kEpiWarp0 + 4 * kPipes * kEpiGroups) * 32;
constexpr int kTileCols = 124;                  // new grid columns per tile (4 quarters x 31; one more is shared)
constexpr int kTapBytes = 64 * 128;             // one filter row's (dx, o) x 64 fp16 of four channels
constexpr int kChunkBytes = 3 * kTapBytes;      // of a group of four channels: filter rows dy = 0, 1, 0, so that both orders are there
constexpr int kEntryCols = 64;                  // tensor-memory columns of an entry: two chunks of 64 fp16
constexpr int kRing = 2, kAcc = 2;              // of a pipe: entries and accumulators (64 columns each) in tensor memory
constexpr int kPipeCols = kAcc * 64 + kRing * kEntryCols;
constexpr int kMaxStages = 4;                   // of a pipe
static_assert(kPipes * kPipeCols <= 512 && kIssueWarp0 + kPipes <= kConvWarp0 && kThreads <= 1024, "tensor memory, warps");
// The barriers carry one parity bit, so a waiter must stay within one phase of its barrier: every accumulator has one
// epilogue group, and uses of it follow one another there.
static_assert(kAcc % kEpiGroups == 0, "phases");

struct Conv1Params {
    Conv1Plan pl;
    const uint8_t* obs;
    const int32_t* slots;   // frame of each row in obs, or nullptr: row e is frame e
    int pool;               // frames in obs when slots are given
    int n;
    int tiles;              // ceil(n * Ws / 124)
    bool shared;            // the pipes of a CTA take half of each tile's rows, not half of the stretch
    const float* bias;
    const float* inv_scale;
    __half* out;
    size_t out_row;         // elements of out from one of its grid rows to the next
    int* status;
};

// Frame index of batch row e: e itself, or its slot in the pool.  A slot outside the pool is
// recorded in the status word and frame 0 is read instead (the heads kernel drops that row).
__device__ __forceinline__ size_t frame_of(const Conv1Params& p, int e)
{
    if (!p.slots) return (size_t)e;
    const int sl = p.slots[e];
    if ((unsigned)sl >= (unsigned)p.pool) { atomicCAS(p.status, 0, kStatusBadSlot); return 0; }
    return (size_t)sl;
}

// Four bytes -> four fp16 values without arithmetic: a byte b zero-extended to 16 bits is the fp16
// subnormal b * 2^-24, which the tensor core multiplies exactly; the 2^24 goes into the accumulator scale.
__device__ __forceinline__ void u8x4_to_h4(uint32_t w, uint32_t& lo, uint32_t& hi)
{
    lo = __byte_perm(w, 0u, 0x4140);                    // {b0, 0, b1, 0}
    hi = __byte_perm(w, 0u, 0x4342);                    // {b2, 0, b3, 0}
}

// A pipe's walk over its output rows, a tile at a time.
struct Portions {
    int H, half, left, next_y;          // output rows of a tile; which half of them to take, or -1; rows not reached, and where they start
    int tile, y, cnt;                   // the pipe's rows y .. y + cnt - 1 of the tile
    // `rows` rows from row r0 of the line on
    __device__ __forceinline__ Portions(int H, int half, int r0, int rows) : H(H), half(half), left(rows), next_y(r0 % H), tile(r0 / H - 1), y(0), cnt(0) { }
    __device__ __forceinline__ bool next()
    {
        while (left > 0) {
            const int c = min(left, H - next_y), first = (c + 1) / 2;
            ++tile;
            y = half == 1 ? next_y + first : next_y;
            cnt = half < 0 ? c : half ? c - first : first;
            left -= c;
            next_y = 0;
            if (cnt > 0) return true;
        }
        return false;
    }
};

// CG: groups of four channels.  WC: the frame width when known at compile time (the converter's loads then
// use immediate offsets), 0 = any.
template <int CG, int WC>
__global__ void __launch_bounds__(kThreads)
conv1_march_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const Conv1Params p)
{
    const Conv1Plan& pl = p.pl;
    constexpr int RE = CG == 1 ? 2 : 1;                // grid rows of an entry
    constexpr int EPR = CG == 4 ? 2 : 1;               // entries of a grid row
    const int W = WC ? WC : pl.W;
    extern __shared__ uint8_t smem_raw[];
    // the filter's barrier, then each pipe's: staged entries, entries in tensor memory, accumulators; full and empty
    constexpr int kPipeBars = 2 * (kMaxStages + kRing + kAcc);
    __shared__ uint64_t bars[1 + kPipes * kPipeBars];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) float s_bias[32];
    volatile int* abortp = &abort_flag;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
    constexpr int w_bytes = CG * kChunkBytes;
    const int NS = pl.stages, Ws = WC ? WC / 4 : pl.Ws, pitch = WC ? 128 * (WC / 4) : pl.env_pitch;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this warp's pipe, and its walk over the pipe's output rows
    const int pipe = warp < kConvWarp0 ? warp % kPipes : warp < kEpiWarp0 ? (warp - kConvWarp0) >> 2 : (warp - kEpiWarp0) / (4 * kEpiGroups);
    const int share = p.tiles * pl.H1 / (int)gridDim.x, extra = p.tiles * pl.H1 - share * (int)gridDim.x;
    const int r0 = (int)blockIdx.x * share + min((int)blockIdx.x, extra), rows = share + ((int)blockIdx.x < extra), mid = p.shared ? 0 : (rows + 1) / 2;
    Portions at(pl.H1, p.shared ? pipe : -1, r0 + (pipe ? mid : 0), p.shared ? rows : pipe ? rows - mid : mid);
    auto entries_of = [](int cnt) { return RE == 2 ? (cnt + 2) / 2 : (cnt + 1) * EPR; };   // of cnt output rows of a tile
    uint64_t *w_bar = bars, *u8_full = bars + 1 + pipe * kPipeBars, *u8_empty = u8_full + kMaxStages, *a_full = u8_empty + kMaxStages,
             *a_empty = a_full + kRing, *d_full = a_empty + kRing, *d_empty = d_full + kAcc;

    // The prologue is on the step's critical path: this CTA gets the SM when the previous kernel's last one leaves it.
    if (warp == 0) {
        for (int i = lane; i < 1 + kPipes * kPipeBars; i += 32) {
            const int j = i ? (i - 1) % kPipeBars : 0;
            mbar_init(&bars[i], i == 0 ? 1 : j < kMaxStages ? kLoadWarps : j < 2 * kMaxStages + kRing ? 4
                                                                          : j < 2 * kMaxStages + 2 * kRing + kAcc ? 1 : 4);
        }
        fence_barrier_init();
        __syncwarp();
        if (lane == 0) {                                 // the filter: not the previous kernel's, see `dependent`
            mbar_arrive_expect_tx(w_bar, (uint32_t)w_bytes);
            for (int g = 0; g < CG; ++g)
                for (int j = 0; j < 3; ++j) tma_load_2d(sm + g * kChunkBytes + j * kTapBytes, &tmW, g * 64, (j & 1) * 64, w_bar);
        }
    } else if (warp == 1) {
        tmem_alloc(&tmem_slot, 512);
    } else if (warp == 2 && lane == 0) {
        abort_flag = 0;
        tma_prefetch_desc(&tmX);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_d = tmem_slot + pipe * kPipeCols, tmem_a = tmem_d + kAcc * 64;
    pdl_wait();
    pdl_trigger();

    if (warp < kIssueWarp0) {
        // ---- staging: one box per environment the tile touches; warp l takes the tile's l-th, (l + kLoadWarps)-th, ...
        const int l = warp / kPipes;
        uint8_t* stages = sm + w_bytes + pipe * NS * pl.stage_bytes + l * pitch;
        int st = 0;
        uint32_t ph = 1;
        bool alive = true;
        while (alive && at.next()) {
            const int entries = entries_of(at.cnt);
            const int e_first = (at.tile * kTileCols) / Ws, envs = min((at.tile * kTileCols + kTileCols) / Ws, p.n - 1) - e_first + 1;
            const int mine = (envs - l + kLoadWarps - 1) / kLoadWarps;               // boxes of this warp: lane i knows the i-th one's frame
            const int frame = lane < mine ? (int)frame_of(p, e_first + l + lane * kLoadWarps) : 0;
            for (int k = 0; k < entries; ++k) {
                if (!mbar_wait_warp(&u8_empty[st], ph, abortp, p.status, 31)) { alive = false; break; }
                uint8_t* dst = stages + st * pl.stage_bytes;
                if (lane == 0) mbar_arrive_expect_tx(&u8_full[st], (uint32_t)(mine * pl.env_pitch));
                for (int i = 0; i < mine; ++i, dst += kLoadWarps * pitch) {
                    const int f = __shfl_sync(0xffffffffu, frame, i);
                    if (lane == 0) tma_load_4d(dst, &tmX, 0, at.y + k * RE / EPR, (k % EPR) * 8, f, &u8_full[st]);
                }
                if (++st == NS) { st = 0; ph ^= 1u; }
            }
        }
    } else if (warp < kIssueWarp0 + kPipes) {
        // ---- MMA issue, entry by entry
        if (elect_one()) {
            constexpr uint32_t id64 = instr_desc_f16(0, 128, 64), id128 = instr_desc_f16(0, 128, 128);
            const uint64_t bdesc = smem_desc_sw128(base);
            int k = 0, ke = 0, c0 = 0;                        // entry of the pipe / of the portion; output rows before the portion
            bool alive = at.next() && mbar_wait(w_bar, 0, abortp, p.status, 32), there = false;
            int cnt = at.cnt, entries = entries_of(cnt);
            while (alive) {
                const int s = k % kRing;
                if (!there && !mbar_wait(&a_full[s], (uint32_t)(k / kRing) & 1u, abortp, p.status, 34)) break;
                tc_fence_after();
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {              // chunks of 64 K values
                    const int i = RE == 2 ? 2 * ke + hf : ke / EPR;                // grid row of the portion
                    const int cg = CG == 1 ? 0 : CG == 2 ? hf : (ke % EPR) * 2 + hf;
                    const bool lo = i > 0 && i <= cnt, hi = i < cnt;               // feeds output rows i - 1 (dy = 1), i (dy = 0)
                    const int c = c0 + i, s0 = c % kAcc;
                    const uint32_t a = tmem_a + s * kEntryCols + hf * 32, d0 = tmem_d + s0 * 64, d1 = tmem_d + (s0 ^ 1) * 64;
                    const uint64_t b0 = bdesc + (uint32_t)(cg * (kChunkBytes >> 4)), b1 = b0 + (kTapBytes >> 4);
                    if (lo && hi && cg > 0) {                 // accumulators in the order (dy = 0, dy = 1) or the other way round
                        const uint64_t b = s0 ? b1 : b0;
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) mma_f16_ts(tmem_d, a + 8 * kk, b + 2 * kk, id128, 1);
                    } else {
                        // output row i starts with chunk 0: row i - 1 first, while output row i - 2 is still being drained
                        if (lo) {
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) mma_f16_ts(d1, a + 8 * kk, b1 + 2 * kk, id64, 1);
                            if (cg == CG - 1) mma_commit(&d_full[s0 ^ 1]);
                        }
                        if (hi) {
                            if (cg == 0 && !mbar_wait(&d_empty[s0], ((uint32_t)(c / kAcc) & 1u) ^ 1u, abortp, p.status, 33)) { alive = false; break; }
                            tc_fence_after();
                            mma_f16_ts(d0, a, b0, id64, cg != 0);
#pragma unroll
                            for (int kk = 1; kk < 4; ++kk) mma_f16_ts(d0, a + 8 * kk, b0 + 2 * kk, id64, 1);
                        }
                    }
                    if (lo && hi && cg > 0 && cg == CG - 1) mma_commit(&d_full[s0 ^ 1]);
                    if (hf == 0) there = mbar_test(&a_full[(k + 1) % kRing], (uint32_t)((k + 1) / kRing) & 1u);
                }
                if (!alive) break;
                mma_commit(&a_empty[s]);
                ++k;
                if (++ke == entries) { ke = 0; c0 += cnt; alive = at.next(); cnt = at.cnt; entries = entries_of(cnt); }
            }
        }
    } else if (warp >= kConvWarp0 && warp < kEpiWarp0) {
        // ---- convert: thread = grid column q of the tile
        const int qq = warp & 3;
        const uint32_t st_addr = tmem_a + ((uint32_t)(qq * 32) << 16);
        const uint8_t* stages = sm + w_bytes + pipe * NS * pl.stage_bytes;
        int k = 0, st = 0;
        uint32_t ph = 0;
        bool alive = true;
        while (alive && at.next()) {
            const int entries = entries_of(at.cnt);
            const int q = at.tile * kTileCols + 31 * qq + lane, e = q / Ws, X = q - e * Ws, e_first = (at.tile * kTileCols) / Ws;
            // columns past the end of the batch read the start of the entry: their results are never stored
            const int off = e < p.n ? (e - e_first) * pitch + 4 * X : 0;
            for (int ke = 0; ke < entries; ++ke, ++k) {
                const int s = k % kRing;
                const uint8_t* src = stages + st * pl.stage_bytes + off;
                if (!mbar_wait_warp(&u8_full[st], ph, abortp, p.status, 35)) { alive = false; break; }
                uint32_t v[32];
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int uy = 0; uy < 4; ++uy)
                            u8x4_to_h4(*reinterpret_cast<const uint32_t*>(src + (RE == 2 ? (c * 2 + hf) * 4 + uy : (hf * 4 + c) * 4 + uy) * W),
                                       v[c * 8 + uy * 2], v[c * 8 + uy * 2 + 1]);
                    if (hf == 0) {
                        if (!mbar_wait_warp(&a_empty[s], ((uint32_t)(k / kRing) & 1u) ^ 1u, abortp, p.status, 36)) { alive = false; break; }
                        tc_fence_after();
                    } else {
                        __syncwarp();                    // the staged bytes are in registers
                        if (lane == 0) mbar_arrive(&u8_empty[st]);
                    }
                    tmem_st_32x32(st_addr + s * kEntryCols + hf * 32, v);
                }
                if (!alive) break;
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&a_full[s]);
                if (++st == NS) { st = 0; ph ^= 1u; }
            }
        }
    } else if (warp >= kEpiWarp0) {
        // ---- epilogue: group g drains output rows g, g + kEpiGroups, ... of the pipe; warp quarter = TMEM lane quarter
        const int g = ((warp - kEpiWarp0) >> 2) % kEpiGroups, qq = warp & 3;
        const float inv = *p.inv_scale;
        s_bias[lane] = p.bias[lane];                    // every epilogue warp writes the same
        __syncwarp();
        int c = g, c0 = 0;                              // output row of the pipe; how many before the portion
        bool alive = true;
        while (alive && at.next()) {
            const int q = at.tile * kTileCols + 31 * qq + lane, e = q / Ws, X = q - e * Ws;
            const bool valid = lane < 31 && e < p.n && X < pl.W1;
            __half* dst0 = p.out + ((size_t)e * pl.W1s + (X >> 1)) * 128 + (X & 1) * 32;
            for (; c < c0 + at.cnt; c += kEpiGroups) {
                const int y = at.y + c - c0;
                const int acc = c % kAcc;
                __half* dst = dst0 + (size_t)(y >> 1) * p.out_row + (y & 1) * 64;
                const uint32_t taddr = tmem_d + acc * 64 + ((uint32_t)(qq * 32) << 16);
                if (!mbar_wait_warp(&d_full[acc], (uint32_t)(c / kAcc) & 1u, abortp, p.status, 37)) { alive = false; break; }
                tc_fence_after();
#pragma unroll
                for (int j = 0; j < 32; j += 16) {          // sixteen output channels a time: 64 registers a thread
                    uint32_t v0[16], v1[16], pk[8];
                    tmem_ld_32x16(taddr + j, v0);           // dx = 0 part of this column's output
                    tmem_ld_32x16(taddr + 32 + j, v1);      // dx = 1 part of the output one column to the left
                    tmem_ld_wait();
                    if (j == 16) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&d_empty[acc]);
                    }
#pragma unroll
                    for (int hh = 0; hh < 8; ++hh) {
                        const int o = 2 * hh;
                        float a0 = __uint_as_float(v0[o]), a1 = __uint_as_float(v0[o + 1]);
                        add2(a0, a1, __shfl_down_sync(0xffffffffu, __uint_as_float(v1[o]), 1),
                             __shfl_down_sync(0xffffffffu, __uint_as_float(v1[o + 1]), 1));
                        fma2(a0, a1, inv, s_bias[j + o], s_bias[j + o + 1]);
                        pk[hh] = relu_pack_h2(a0, a1);
                    }
                    if (valid)
                        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                                     ::"l"(dst + j), "r"(pk[0]), "r"(pk[1]), "r"(pk[2]), "r"(pk[3]), "r"(pk[4]), "r"(pk[5]),
                                       "r"(pk[6]), "r"(pk[7]) : "memory");
                }
            }
            c0 += at.cnt;
        }
    }
    if (*abortp) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_slot, 512);
}

template <int CG, int WC>
hts_status launch_variant(const CUtensorMap& weight_map, const CUtensorMap& frame_map, const Conv1Params& p, int grid, bool dependent, cudaStream_t s)
{
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(conv1_march_kernel<CG, WC>, allowed));
    // every kernel of the step asks for the largest shared-memory carve-out, so that the SMs are not
    // re-partitioned between consecutive kernels
    HTS_CUDA(launch_chained(dependent, conv1_march_kernel<CG, WC>, dim3(grid), dim3(kThreads),
                            (size_t)(1024 + CG * kChunkBytes + kPipes * p.pl.stages * p.pl.stage_bytes), s, weight_map, frame_map, p));
    note_launch();
    return HTS_OK;
}

}  // namespace

bool conv1_plan(const Geometry& g, Conv1Plan* pl)
{
    if (g.H % 4 || g.W % 4 || (g.C != 4 && g.C != 8 && g.C != 16) || g.W > 1024) return false;
    pl->C = g.C; pl->H = g.H; pl->W = g.W;
    pl->Hs = g.H / 4; pl->Ws = g.W / 4;
    pl->H1 = pl->Hs - 1; pl->W1 = pl->Ws - 1;
    if (pl->H1 != g.H1 || pl->W1 != g.W1 || pl->Ws < 2 || pl->H1 < 1) return false;
    pl->env_pitch = 128 * pl->Ws;                        // two rows of four channels or one of eight
    pl->stage_bytes = (kTileCols / pl->Ws + 2) * pl->env_pitch;     // the most environments a tile can touch
    pl->stages = (226 * 1024 - 1024 - g.C / 4 * kChunkBytes) / (kPipes * pl->stage_bytes);
    if (pl->stages > kMaxStages) pl->stages = kMaxStages;
    pl->H1s = (pl->H1 + 1) / 2; pl->W1s = (pl->W1 + 1) / 2; pl->P1s = pl->H1s * pl->W1s;
    return true;
}

hts_status conv1_launch(const Conv1Plan& pl, const CUtensorMap& weight_map, Conv1MapCache& maps, const uint8_t* obs,
                        const Indexing& ix, int n, const float* bias, const float* inv_scale, __half* out, int env_rows, int* status,
                        bool dependent, cudaStream_t s)
{
    const int sm_count = device_sm_count(device_slot());
    const long cols = (long)n * pl.Ws;
    if (cols >= (1L << 31) - 256) return HTS_ERR_INVALID_ARG;
    // the tensor map over this frame buffer (dense: n frames; gathered: the whole pool)
    const int frames = ix.slots ? ix.pool : n;
    int slot = -1;
    for (int i = 0; i < Conv1MapCache::kEntries; ++i)
        if (maps.ptr[i] == obs && maps.frames[i] == frames) { slot = i; break; }
    if (slot < 0) {
        slot = maps.next;
        maps.next = (maps.next + 1) % Conv1MapCache::kEntries;
        if (!make_frames_map(&maps.map[slot], obs, pl.W, pl.H, pl.C, (uint64_t)frames, pl.C == 4 ? 2 : 1, pl.C == 4 ? 4 : 8)) {
            maps.ptr[slot] = nullptr;
            return HTS_ERR_CUDA;
        }
        maps.ptr[slot] = obs; maps.frames[slot] = frames;
    }
    Conv1Params p{};
    p.pl = pl; p.obs = obs; p.slots = ix.slots; p.pool = ix.pool; p.n = n;
    p.tiles = (int)((cols + kTileCols - 1) / kTileCols);
    p.bias = bias; p.inv_scale = inv_scale; p.out = out; p.out_row = (size_t)env_rows * pl.W1s * 128; p.status = status;
    const int rows = p.tiles * pl.H1, grid = rows < sm_count ? rows : sm_count;
    p.shared = pl.C == 4 && p.tiles >= 4 * grid;
    if (pl.C == 4) {
        if (pl.W == 84) return launch_variant<1, 84>(weight_map, maps.map[slot], p, grid, dependent, s);
        return launch_variant<1, 0>(weight_map, maps.map[slot], p, grid, dependent, s);
    }
    if (pl.C == 8 && pl.W == 84) return launch_variant<2, 84>(weight_map, maps.map[slot], p, grid, dependent, s);
    if (pl.C == 8) return launch_variant<2, 0>(weight_map, maps.map[slot], p, grid, dependent, s);
    if (pl.W == 96) return launch_variant<4, 96>(weight_map, maps.map[slot], p, grid, dependent, s);
    return launch_variant<4, 0>(weight_map, maps.map[slot], p, grid, dependent, s);
}

}  // namespace hts
