// Dense layer for batches of several row tiles: [n, F] x [512, F]^T on pairs of SMs (tcgen05, cta_group::2).
//
// The result is defined as  h = relu(bias + p_0 + p_1 + ... + p_{S-1}),  p_s = inv * (sum over the K chunks of range s,
// accumulated in tensor memory in chunk order), the p_s added in index order in fp32.  S is a constant of the geometry, so
// the bits do not depend on the batch.
//
// What bounds it is the copy of operands into the SMs: the L2 delivers about 90 bytes per ns to one SM (measured here as 32 KB
// every 0.36 us), and a 128 x 128 tile per SM needs 128 bytes per tensor clock.  A pair of SMs holds a tile of 256 rows and BN
// columns; each of the two copies its own 128 rows of activations and half of the weight rows, and the tensor cores read the
// other half from the partner: 96 (BN = 128) or 64 (BN = 256) bytes per tensor clock.  With all ranges of a tile on one pair, the
// hidden layer leaves the chip once (2 KB per observation) and the pipeline never drains between ranges.  Against 128 x 128
// tiles on single SMs: n = 8192 45 -> 25 us (18 of them copies), a step of 2048 observations 83 -> 72 us, of 4096 124 -> 115.
//
// Where there are fewer tiles than pairs of SMs, the ranges of a tile are dealt to several pairs.  The first keeps the running
// sum of its ranges, the others hand on each range by itself (the order of the additions is fixed), and the heads kernel adds
// what is left: 4 planes instead of 7 at two pairs per tile.  While one range per pair fits the SMs (n <= 1280 for seven
// ranges), 256-column tiles have the least to copy after the previous kernel (112 KB per SM; the weights are asked for
// before it ends) and all seven planes are handed on: step of 1024 observations 47.5 us, with two ranges a pair and 128
// columns 49.4, with a 128 x 128 tile and one range per CTA 48.5.
//
// Roles in each CTA: one thread copies, one thread of the pair's first CTA issues all MMAs, eight warps drain two alternating
// accumulators.  All waits are bounded.
#include "fc_tc.cuh"
#include "tc_ptx.cuh"

namespace hts {
using namespace tc;

namespace {

constexpr int kThreads = 320;                   // warp 0 copies, warp 1 issues, warps 2..9 epilogue (two per lane quarter)
constexpr int kChunk = 64;                      // 16-bit columns of a K chunk: one 128-byte swizzle row
constexpr int kABytes = 128 * 128;
constexpr int kTurn = 32 * 36;                  // floats of a warp's transposing buffer

template <int BN> struct PairShape {
    static constexpr int kBBytes = BN / 2 * 128;                // this CTA's half of the weight rows
    static constexpr int kStage = kABytes + kBBytes;
    static constexpr int kTurnBytes = 8 * kTurn * 4;
    static constexpr int kStages = (226 * 1024 - 1024 - kTurnBytes) / kStage;
    static constexpr int kSmem = 1024 + kStages * kStage + kTurnBytes;
};

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address of a shared variable in the pair's first CTA
__device__ __forceinline__ uint32_t in_first(const void* p)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
    return r;
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// into this CTA's shared memory, completion on a barrier of either CTA of the pair
__device__ __forceinline__ void tma_load_2d_pair(void* smem_dst, const CUtensorMap* map, int x, int y, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(smem_u32(smem_dst)), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ void mma_f16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// arrives at the barrier in both CTAs
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}

// ONE: each pair has one range and hands it on as it is.  <256, true> takes 64 registers and spills 16 bytes.
template <int BN, bool ONE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads)
fc_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const FcPairParams p)
{
    using S = PairShape<BN>;
    constexpr int NST = S::kStages, HALF = BN / 2;
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bars[2 * NST + 4];
    uint64_t *full_bar = bars, *empty_bar = bars + NST, *acc_full = empty_bar + NST, *acc_empty = acc_full + 2;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ float s_bias[BN];
    volatile int* abortp = &abort_flag;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;      // the same offset in both CTAs
    uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank();
    const int m0 = blockIdx.x * 128, n0 = blockIdx.y * BN;           // blockIdx.x = 2 * tile + rank
    const int s0 = blockIdx.z * p.group, ns = min(p.group, p.splits - s0);
    const int k0 = s0 * p.cps, chunks = ns * p.cps;

    if (warp == 0) {
        if (lane < 2 * NST + 4) mbar_init(&bars[lane], lane < 2 * NST + 2 ? 1 : 16);
        fence_barrier_init();
    } else if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(2 * BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else if (warp == 2 && lane == 0) {
        abort_flag = 0;
        tma_prefetch_desc(&tmA);
    }
    static_assert(2 * NST + 4 <= 32, "a lane initialises one barrier");
    tc_fence_before();
    cluster_sync();                                      // of both CTAs' threads: the partner's barriers exist
    tc_fence_after();
    const uint32_t tmem_d = tmem_slot;

    // Stage s of either CTA completes the first CTA's barrier, which expects both CTAs' bytes.
    auto load_b = [&](int kc, int st) {
        uint8_t* dst = sm + st * S::kStage + kABytes;
        const uint32_t bar = in_first(&full_bar[st]);
        if (rank == 0) mbar_arrive_expect_tx(&full_bar[st], 2 * S::kStage);
#pragma unroll
        for (int i = 0; i < HALF / 64; ++i) tma_load_2d_pair(dst + i * 8192, &tmB, (k0 + kc) * kChunk, n0 + rank * HALF + 64 * i, bar);
    };
    if (warp == 0 && lane == 0)                          // the weights do not depend on the previous kernel
        for (int kc = 0; kc < NST && kc < chunks; ++kc) load_b(kc, kc);
    pdl_wait();
    pdl_trigger();

    if (warp == 0) {
        if (lane == 0) {
            for (int kc = 0; kc < chunks; ++kc) {
                const int st = kc % NST;
                if (kc >= NST) {
                    if (!mbar_wait(&empty_bar[st], ((uint32_t)(kc / NST) & 1u) ^ 1u, abortp, p.status, 51)) break;
                    load_b(kc, st);
                }
                tma_load_2d_pair(sm + st * S::kStage, &tmA, (k0 + kc) * kChunk, p.row0 + m0, in_first(&full_bar[st]));
            }
        }
    } else if (warp == 1) {
        if (rank == 0 && elect_one()) {
            constexpr uint32_t idesc = instr_desc_f16(0, 256, BN);
            int kc = 0;
            bool alive = true;
            for (int sp = 0; alive && sp < ns; ++sp) {
                const int acc = sp & 1;
                if (!mbar_wait(&acc_empty[acc], ((uint32_t)(sp >> 1) & 1u) ^ 1u, abortp, p.status, 52)) break;
                tc_fence_after();
                for (int c = 0; c < p.cps; ++c, ++kc) {
                    const int st = kc % NST;
                    if (!mbar_wait(&full_bar[st], (uint32_t)(kc / NST) & 1u, abortp, p.status, 53)) { alive = false; break; }
                    tc_fence_after();
                    const uint32_t a_addr = base + st * S::kStage;
                    const uint64_t adesc = smem_desc_sw128(a_addr), bdesc = smem_desc_sw128(a_addr + kABytes);
#pragma unroll
                    for (int k = 0; k < kChunk / 16; ++k)
                        mma_f16_pair(tmem_d + acc * BN, adesc + 2 * k, bdesc + 2 * k, idesc, (c | k) != 0);
                    mma_commit_pair(&empty_bar[st]);
                }
                if (alive) mma_commit_pair(&acc_full[acc]);
            }
        }
    } else {
        // epilogue warps 2..9: lane quarter warp % 4, columns [HALF half, HALF half + HALF) of the tile
        const int q = warp & 3, half = (warp - 2) >> 2;
        const float inv = *p.inv_scale;
        if constexpr (!ONE) {                            // the two to four warps that share a column write the same
            for (int i = lane; i < HALF; i += 32) s_bias[half * HALF + i] = p.bias[n0 + half * HALF + i];
            __syncwarp();
        }
        const bool running = !ONE && (BN == 256 || blockIdx.z == 0);      // a wide tile has one range or all of them
        float* turn = reinterpret_cast<float*>(sm + NST * S::kStage) + (warp - 2) * kTurn;
        const int row0 = m0 + q * 32, col0 = n0 + half * HALF, rl = lane >> 3, c4 = (lane & 7) * 4;
        // a row per thread, turned through shared memory so that eight lanes write one full 128-byte line
        auto store32 = [&](float* out, int c, const float (&v)[32]) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) *reinterpret_cast<float4*>(turn + lane * 36 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int rr = 4 * i + rl;
                const float4 val = *reinterpret_cast<const float4*>(turn + rr * 36 + c4);
                if (row0 + rr < p.n) *reinterpret_cast<float4*>(out + (size_t)(row0 + rr) * 512 + col0 + c + c4) = val;
            }
            __syncwarp();
        };
        float sum[ONE ? 1 : HALF];
        bool ok = true;
        for (int sp = 0; ok && sp < ns; ++sp) {
            const int acc = sp & 1;
            ok = mbar_wait_warp(&acc_full[acc], (uint32_t)(sp >> 1) & 1u, abortp, p.status, 54);
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = tmem_d + acc * BN + half * HALF + ((uint32_t)(q * 32) << 16);
#pragma unroll
            for (int c = 0; c < HALF; c += 32) {
                float t[32];
#pragma unroll
                for (int hf = 0; hf < 32; hf += 16) {     // sixteen columns a time: with 32, 256-column tiles spill
                    uint32_t v[16];
                    tmem_ld_32x16(taddr + c + hf, v);
                    tmem_ld_wait();
                    if (c + hf + 16 == HALF) {            // the accumulator is in registers: hand it back
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0 && sp + 2 < ns) arrive_cluster(in_first(&acc_empty[acc]));      // what is waited for, and no more
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float ps = __fmul_rn(__uint_as_float(v[j]), inv);
                        if constexpr (!ONE) {
                            if (running) sum[c + hf + j] = sp == 0 ? ps : __fadd_rn(sum[c + hf + j], ps);      // in index order, as the heads kernel adds planes
                            else t[hf + j] = ps;
                        } else t[hf + j] = ps;
                    }
                }
                if (!running) store32(p.planes + (size_t)(s0 + sp - p.group + 1) * p.plane_stride, c, t);
            }
        }
        if constexpr (!ONE) if (ok && running) {
            const bool last = BN == 256 || ns == p.splits;
#pragma unroll
            for (int c = 0; c < HALF; c += 32) {
                float t[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) t[j] = last ? fmaxf(__fadd_rn(sum[c + j], s_bias[half * HALF + c + j]), 0.f) : sum[c + j];
                store32(last ? p.h : p.planes, c, t);
            }
        }
    }
    if (*abortp) {                                       // give copies still in flight time to land
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }
    }
    tc_fence_before();
    __syncthreads();
    // neither CTA leaves while the other's MMAs need its memory; stores need not have arrived for that
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(2 * BN) : "memory");
}

template <int BN, bool ONE>
hts_status launch(const CUtensorMap& a, const CUtensorMap& b, const FcPairParams& p, cudaStream_t s)
{
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(fc_pair_kernel<BN, ONE>, allowed));
    const dim3 grid(2 * ((p.n + 255) / 256), 512 / BN, (p.splits + p.group - 1) / p.group);
    HTS_CUDA(launch_pdl(fc_pair_kernel<BN, ONE>, grid, dim3(kThreads), (size_t)PairShape<BN>::kSmem, s, a, b, p));
    note_launch();
    return HTS_OK;
}

}  // namespace

FcPairPlan fc_pair_plan(int n, int splits)
{
    const int pairs = device_sm_count(device_slot()) / 2, m_tiles = (n + 255) / 256;
    if (splits > 1 && 2 * m_tiles * splits <= pairs) return {true, 1, splits};
    const int tiles = 4 * m_tiles;
    if (tiles > pairs) return {true, splits, 1};
    const int groups = pairs / tiles < splits ? pairs / tiles : splits, group = (splits + groups - 1) / groups;
    return {false, group, 1 + splits - group};
}

hts_status fc_pair_launch(const CUtensorMap& act_map, const CUtensorMap& weight_map, const FcPairParams& p, bool wide, cudaStream_t s)
{
    if (!wide) return launch<128, false>(act_map, weight_map, p, s);
    return p.group < p.splits ? launch<256, true>(act_map, weight_map, p, s) : launch<256, false>(act_map, weight_map, p, s);
}

}  // namespace hts
