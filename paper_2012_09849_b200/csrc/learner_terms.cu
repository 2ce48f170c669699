// Sample means over the stored transitions that the learner's objectives are built from:
//   hts_a2c_terms  Section 3: the policy term of Eq. 4, (1/|D|) sum log pi(a|s) (R - V), the value loss
//                  J_V = (1/|D|) sum (R - V)^2 and the mean entropy;
//   hts_ppo_terms  the clipped surrogate of proximal policy optimisation (Schulman et al. 2017, Eq. 7), the
//                  algorithm the football runs of Section 5 use, with the same value loss and entropy.
//
// HBM-bound (16 to 28 bytes per transition).  Each block sums a contiguous range in double precision in a
// fixed order (thread-strided float4 loads, shuffle tree, warp order), writes its partial and takes a
// ticket; the block that draws the last ticket adds the partials in a fixed order.  The grid is a
// function of the count alone; the order of the sums depends besides on whether the inputs are 16-byte aligned and, for
// standardised terms, on whether the device has room for a cluster.  It depends neither on timing nor on the device's load.
#include <cmath>
#include "common.cuh"
#include "tc_ptx.cuh"

namespace hts {
namespace {

constexpr int kBlocksMax = 2048;
constexpr int kThreads = 256;
constexpr int kPerThread = 8;             // elements a thread covers before another block is worth its launch
constexpr int kMaxSums = 4;

// Partials, the ticket counter and the advantage statistics live in the library image: calls on one device
// must not overlap.
__device__ double g_partial[kBlocksMax][kMaxSums];
__device__ unsigned int g_ticket;
__device__ double g_adv_stats[2];         // mean and 1 / (std + 1e-8) of the advantages (hts_ppo_terms)

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
    return v;
}

// How a kernel of sums follows the one before it.  Not Alone: that one is a kernel of sums as well, over the same inputs.  It has
// waited for whatever wrote them, so the first loads (two groups of a thread, all that it has up to kThreads * kPerThread elements
// to a block) need not wait for it: they are under way while it runs.  Its 48 registers of inputs decide how many blocks an SM
// holds, so there are two forms.  Standardised means, us, inputs not in cache (both launches):
//   transitions            131072  300000  600000 | 640000  768000  900000  1000000  2000000  4000000  16000000
//   Alone, 70 registers       9.6    12.3    14.1 |   13.7    16.2    15.4     20.2     29.0     47.7     116.2
//   EarlyTwo, 102             8.3     9.7    11.7 |   13.8    16.3    16.0     18.1     28.5     50.3
//   EarlyThree, 80            8.7     9.9    12.3 |   12.6    14.9    13.9     17.7     26.6     43.8      96.8
// EarlyTwo while all blocks are on the device at two per SM (606208 transitions on 148 SMs); above that, a third block per SM saves
// a wave (up to 909312) or covers more latency.
enum class Form { Alone, EarlyTwo, EarlyThree };

// An Op names NS sums, how four consecutive elements (float4 group q) or one element i add to them, whether
// its arrays allow float4 loads, and what the last block does with the totals.
template <class Op, Form FORM>
__global__ void __launch_bounds__(kThreads, FORM == Form::EarlyThree ? 3 : 0)
sums_kernel(const Op op, long long count, long long per_block)
{
    constexpr bool CHAINED = FORM != Form::Alone;
    constexpr int NS = Op::NS;
    __shared__ double s_part[kThreads / 32][NS];
    __shared__ bool s_last;
    if constexpr (!CHAINED) { pdl_wait(); pdl_trigger(); }                // the partials, the ticket and the inputs are the previous kernel's
    const long long lo = (long long)blockIdx.x * per_block;               // per_block is a multiple of 4
    long long hi = lo + per_block; hi = hi > count ? count : hi;
    double acc[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) acc[k] = 0.0;
    if (op.aligned16()) {
        const long long q_lo = lo >> 2, q_hi = hi >> 2;                    // whole float4 groups of the range
        long long q = q_lo + threadIdx.x;
        if constexpr (CHAINED) {
            static_assert(kPerThread == 8, "two groups are all that a thread of an EarlyTwo block has");
            typename Op::Quad g[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) if (q + u * kThreads < q_hi) g[u] = op.load4(q + u * kThreads);
            pdl_wait();
            pdl_trigger();
#pragma unroll
            for (int u = 0; u < 2; ++u) if (q + u * kThreads < q_hi) op.add4(g[u], acc);
            q += 2 * kThreads;
        }
        if constexpr (FORM != Form::EarlyTwo) {
            constexpr int U = FORM == Form::Alone ? 4 : 2;                 // groups per array in flight per thread
            for (; q + (U - 1) * kThreads < q_hi; q += U * kThreads) {
                typename Op::Quad g[U];
#pragma unroll
                for (int u = 0; u < U; ++u) g[u] = op.load4(q + u * kThreads);
#pragma unroll
                for (int u = 0; u < U; ++u) op.add4(g[u], acc);
            }
            for (; q < q_hi; q += kThreads) op.add4(op.load4(q), acc);
        }
        for (long long i = (q_hi << 2) + threadIdx.x; i < hi; i += kThreads) op.add1(i, acc);   // the last block's ragged tail
    } else {
        if constexpr (CHAINED) { pdl_wait(); pdl_trigger(); }
        for (long long i = lo + threadIdx.x; i < hi; i += kThreads) op.add1(i, acc);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        acc[k] = warp_sum_d(acc[k]);
        if (lane == 0) s_part[warp][k] = acc[k];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            double a = 0.0;
            for (int w = 0; w < kThreads / 32; ++w) a += s_part[w][k];
            g_partial[blockIdx.x][k] = a;
        }
        __threadfence();
        s_last = atomicAdd(&g_ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last && threadIdx.x < 32) {
        // lane l adds partials l, l + 32, ... in that order, then the lanes are folded by a shuffle tree: an order
        // fixed by the grid size, whatever the arrival order of the blocks
        __threadfence();
        double tot[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) tot[k] = 0.0;
        for (unsigned b = threadIdx.x; b < gridDim.x; b += 32)
#pragma unroll
            for (int k = 0; k < NS; ++k) tot[k] += *(volatile double*)&g_partial[b][k];
#pragma unroll
        for (int k = 0; k < NS; ++k) tot[k] = warp_sum_d(tot[k]);
        if (threadIdx.x == 0) {
            op.finish(tot, count);
            g_ticket = 0;                                                    // ready for the next launch
        }
    }
}

struct SumsGrid { long long blocks, per_block; };
inline SumsGrid sums_grid(long long count)
{
    long long blocks = (count + (long long)kThreads * kPerThread - 1) / ((long long)kThreads * kPerThread);
    if (blocks > kBlocksMax) blocks = kBlocksMax;
    long long per_block = (count + blocks - 1) / blocks;
    per_block = (per_block + 3) / 4 * 4;
    return {(count + per_block - 1) / per_block, per_block};
}

template <Form FORM = Form::Alone, class Op>
hts_status launch_sums(const Op& op, long long count, cudaStream_t s)
{
    const SumsGrid g = sums_grid(count);
    HTS_CUDA(launch_pdl(sums_kernel<Op, FORM>, dim3((unsigned)g.blocks), dim3(kThreads), 0, s, op, count, g.per_block));
    note_launch();
    return HTS_OK;
}

inline bool all_aligned16(std::initializer_list<const void*> ps)
{
    uintptr_t x = 0;
    for (const void* p : ps) x |= (uintptr_t)p;
    return (x & 15u) == 0;
}

struct A2cOp {
    static constexpr int NS = 3;
    const float *logp, *values, *entropy, *returns;
    float* out;
    bool vec;
    struct Quad { float4 l, v, h, r; };
    __device__ bool aligned16() const { return vec; }
    __device__ Quad load4(long long q) const
    {
        return Quad{reinterpret_cast<const float4*>(logp)[q], reinterpret_cast<const float4*>(values)[q],
                    reinterpret_cast<const float4*>(entropy)[q], reinterpret_cast<const float4*>(returns)[q]};
    }
    __device__ static void one(float l, float v, float h, float r, double* acc)
    {
        const double a = (double)r - v;
        acc[0] += (double)l * a; acc[1] += a * a; acc[2] += (double)h;
    }
    __device__ void add4(const Quad& g, double* acc) const
    {
        one(g.l.x, g.v.x, g.h.x, g.r.x, acc); one(g.l.y, g.v.y, g.h.y, g.r.y, acc);
        one(g.l.z, g.v.z, g.h.z, g.r.z, acc); one(g.l.w, g.v.w, g.h.w, g.r.w, acc);
    }
    __device__ void add1(long long i, double* acc) const { one(logp[i], values[i], entropy[i], returns[i], acc); }
    __device__ void finish(const double* tot, long long count) const
    {
        const double inv = 1.0 / (double)count;
        out[0] = (float)(tot[0] * inv); out[1] = (float)(tot[1] * inv); out[2] = (float)(tot[2] * inv);
    }
};

// Mean and 1 / (population std + 1e-8) of the advantages in one pass: sums of a - a_0 and its square in double
// precision (the shift keeps a mean far from zero from cancelling the variance).
struct AdvStatsOp {
    static constexpr int NS = 2;
    const float* adv;
    bool vec;
    using Quad = float4;
    __device__ bool aligned16() const { return vec; }
    __device__ Quad load4(long long q) const { return reinterpret_cast<const float4*>(adv)[q]; }
    __device__ static void one(float a, double first, double* acc) { const double d = (double)a - first; acc[0] += d; acc[1] += d * d; }
    __device__ void add4(const Quad& g, double* acc) const
    {
        const double f = (double)adv[0];
        one(g.x, f, acc); one(g.y, f, acc); one(g.z, f, acc); one(g.w, f, acc);
    }
    __device__ void add1(long long i, double* acc) const { one(adv[i], (double)adv[0], acc); }
    __device__ static void standardise(double sum, double squares, double first, long long count, double* stats)
    {
        const double d = sum / (double)count, var = squares / (double)count - d * d;
        stats[0] = first + d;
        stats[1] = 1.0 / (sqrt(var > 0.0 ? var : 0.0) + 1e-8);
    }
    __device__ void finish(const double* tot, long long count) const { standardise(tot[0], tot[1], (double)adv[0], count, g_adv_stats); }
};

// IN_TURN: an element's sums are finished before the next one's are begun (the compiler otherwise works on all eight of two groups
// at once, 110 registers).
template <bool IN_TURN>
struct PpoOp {
    static constexpr int NS = 4;
    const float *logp_new, *logp_old, *values, *entropy, *adv, *returns;
    float* out;
    double clip;
    bool normalize, vec;
    struct Quad { float4 ln, lo, v, h, a, r; };
    __device__ bool aligned16() const { return vec; }
    __device__ Quad load4(long long q) const
    {
        return Quad{reinterpret_cast<const float4*>(logp_new)[q], reinterpret_cast<const float4*>(logp_old)[q],
                    reinterpret_cast<const float4*>(values)[q], reinterpret_cast<const float4*>(entropy)[q],
                    reinterpret_cast<const float4*>(adv)[q], reinterpret_cast<const float4*>(returns)[q]};
    }
    __device__ void one(float ln, float lo, float v, float h, float a, float r, double mean, double inv_std, double* acc) const
    {
        const double rho = (double)expf(ln - lo);           // fp32 exponential (2 ulp): the fp64 one would bound the kernel
        const double adv_n = ((double)a - mean) * inv_std;
        const double clipped = fmin(fmax(rho, 1.0 - clip), 1.0 + clip);
        acc[0] += fmin(rho * adv_n, clipped * adv_n);
        const double d = (double)r - v;
        acc[1] += d * d;
        acc[2] += (double)h;
        acc[3] += fabs(rho - 1.0) > clip ? 1.0 : 0.0;
    }
    __device__ static void in_turn(float& ln, float& lo, float& v, float& a, float& r, double* acc)
    {
        if constexpr (IN_TURN)
            asm volatile("" : "+f"(ln), "+f"(lo), "+f"(v), "+f"(a), "+f"(r), "+d"(acc[0]), "+d"(acc[1]), "+d"(acc[2]), "+d"(acc[3]));
    }
    __device__ void add4(Quad g, double m, double is, double* acc) const
    {
        in_turn(g.ln.x, g.lo.x, g.v.x, g.a.x, g.r.x, acc); one(g.ln.x, g.lo.x, g.v.x, g.h.x, g.a.x, g.r.x, m, is, acc);
        in_turn(g.ln.y, g.lo.y, g.v.y, g.a.y, g.r.y, acc); one(g.ln.y, g.lo.y, g.v.y, g.h.y, g.a.y, g.r.y, m, is, acc);
        in_turn(g.ln.z, g.lo.z, g.v.z, g.a.z, g.r.z, acc); one(g.ln.z, g.lo.z, g.v.z, g.h.z, g.a.z, g.r.z, m, is, acc);
        in_turn(g.ln.w, g.lo.w, g.v.w, g.a.w, g.r.w, acc); one(g.ln.w, g.lo.w, g.v.w, g.h.w, g.a.w, g.r.w, m, is, acc);
    }
    __device__ void add1(long long i, double m, double is, double* acc) const
    {
        one(logp_new[i], logp_old[i], values[i], entropy[i], adv[i], returns[i], m, is, acc);
    }
    __device__ void add4(const Quad& g, double* acc) const { add4(g, normalize ? g_adv_stats[0] : 0.0, normalize ? g_adv_stats[1] : 1.0, acc); }
    __device__ void add1(long long i, double* acc) const { add1(i, normalize ? g_adv_stats[0] : 0.0, normalize ? g_adv_stats[1] : 1.0, acc); }
    __device__ void finish(const double* tot, long long count) const
    {
        const double inv = 1.0 / (double)count;
        for (int k = 0; k < 4; ++k) out[k] = (float)(tot[k] * inv);
    }
};

// Standardised terms of few transitions in one launch: a cluster of up to 16 blocks whose shared memory holds all inputs, so that
// the advantages' statistics and the terms are two passes over it, with the blocks' sums exchanged through each other's shared
// memory in between.  The sums' order is fixed by the count; nothing global is written but the results.  Bound: one launch (4.3 us
// for the host, where two take 6.5), then copies into at most 16 SMs and fp64 conversions and sums there.  Standardised means, us, calls in a row:
//   transitions        64   2048  16384  50000  131072  147455
//   two launches     7.67   8.26   8.13   8.52    9.06    9.93
//   one              4.22   4.50   5.30   6.18    7.79    8.39
// so it is taken as long as the inputs fit.  Beside actor steps of 1024 on another stream, which leave few SMs free, the median call
// takes 20, 16, 23, 24, 27 and 26 us (at 147456), two launches 30, 31, 28, 32, 32 and 32; the steps take as long beside either.  512
// transitions to a block (2048: 5.42 at 2048; 256: the same); 256 or 1024 threads: 8.0 and 9.0 at 131072, 4.3 and 5.6 at 2048.  16-byte
// asynchronous copies of the threads instead of bulk copies: 8.2 at 131072.  The terms without the advantages summed while the
// statistics cross the cluster: 8.24 (the ratios pass through shared memory once more).  A cooperative launch of sums_kernel's blocks
// with a barrier across the grid: 8.2 whatever the count, 9.3 at 131072.
constexpr int kClusterMost = 16, kClusterThreads = 512, kClusterHolds = 9216;      // transitions of a block: 24 bytes each
constexpr int kClusterEach = 512;                        // transitions before another block is worth its place
constexpr int kClusterWarps = kClusterThreads / 32;

__device__ __forceinline__ void cluster_started() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    cluster_wait();
}
__device__ __forceinline__ void store_to_rank(double* here, unsigned rank, double v)
{
    uint32_t there;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(tc::smem_u32(here)), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(there), "d"(v) : "memory");
}

__global__ void __launch_bounds__(kClusterThreads, 1) terms_cluster_kernel(const PpoOp<false> op, int count, int per_block, bool lost)
{
    constexpr int NS = PpoOp<false>::NS;
    extern __shared__ __align__(16) float4 s_in[];       // [6][per_block / 4]: advantages first
    __shared__ uint64_t landed[2];                       // advantages; the others
    __shared__ int gave_up;
    __shared__ double s_warp[kClusterWarps][NS], s_stat[kClusterMost][2], s_all[kClusterMost][NS];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned rank = blockIdx.x, ranks = gridDim.x;
    if (tid == 0) {
        tc::mbar_init(landed, 1); tc::mbar_init(landed + 1, 1);
        gave_up = 0;
        tc::fence_barrier_init();
    }
    __syncthreads();
    cluster_started();
    pdl_wait();
    pdl_trigger();
    const int lo = rank * per_block, n = max(0, min(per_block, count - lo)), quads = n >> 2, pitch = per_block >> 2;
    const double first = (double)op.adv[0];
    if (tid == 0 && quads > 0 && !lost) {
        const float* const arrays[6] = {op.adv, op.logp_new, op.logp_old, op.values, op.entropy, op.returns};
        tc::mbar_arrive_expect_tx(landed, quads * 16);
        tc::mbar_arrive_expect_tx(landed + 1, 5 * quads * 16);
#pragma unroll
        for (int a = 0; a < 6; ++a) tc::bulk_load(s_in + a * pitch, arrays[a] + lo, quads * 16, landed + (a > 0));
    }
    // The last block's ragged transitions are read where they are.
    const int i = lo + 4 * quads + tid;
    const bool ragged = tid < (n & 3);
    double st[2] = {0.0, 0.0};
    const long long limit = lost ? 100000 : tc::kWaitLimitTicks;
    auto copied = [&](int a, const float*, int q) { return s_in[a * pitch + q]; };
    // Where copies do not land, a warp reads the same inputs where they are.
    auto global = [&](int, const float* from, int q) { return reinterpret_cast<const float4*>(from + lo)[q]; };
    auto add_stats = [&](auto input) {
        for (int q = tid; q < quads; q += kClusterThreads) {
            const float4 a = input(0, op.adv, q);
            AdvStatsOp::one(a.x, first, st); AdvStatsOp::one(a.y, first, st); AdvStatsOp::one(a.z, first, st); AdvStatsOp::one(a.w, first, st);
        }
    };
    if (quads > 0) {
        if (tc::mbar_wait_warp(landed, 0, &gave_up, nullptr, 0, limit)) add_stats(copied);
        else add_stats(global);
    }
    if (ragged) AdvStatsOp::one(op.adv[i], first, st);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        st[k] = warp_sum_d(st[k]);
        if (lane == 0) s_warp[warp][k] = st[k];
    }
    __syncthreads();
    cluster_wait();                                      // every block has started: its shared memory may be written from here on
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const double v = warp_sum_d(lane < kClusterWarps ? s_warp[lane][k] : 0.0);
            if (lane < ranks) store_to_rank(&s_stat[rank][k], lane, v);
        }
    }
    cluster_sync();
    double stats[2], tot[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) tot[k] = warp_sum_d(lane < ranks ? s_stat[lane][k] : 0.0);
    AdvStatsOp::standardise(tot[0], tot[1], first, count, stats);
    double acc[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) acc[k] = 0.0;
    auto add_terms = [&](auto input) {
        for (int q = tid; q < quads; q += kClusterThreads)
            op.add4(PpoOp<false>::Quad{input(1, op.logp_new, q), input(2, op.logp_old, q), input(3, op.values, q), input(4, op.entropy, q),
                                       input(0, op.adv, q), input(5, op.returns, q)}, stats[0], stats[1], acc);
    };
    if (quads > 0) {
        if (tc::mbar_wait_warp(landed, 0, &gave_up, nullptr, 0, limit) && tc::mbar_wait_warp(landed + 1, 0, &gave_up, nullptr, 0, limit)) add_terms(copied);
        else add_terms(global);
    }
    if (ragged) op.add1(i, stats[0], stats[1], acc);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        acc[k] = warp_sum_d(acc[k]);
        if (lane == 0) s_warp[warp][k] = acc[k];         // the statistics in it were read before the cluster's barrier
    }
    __syncthreads();
    if (warp == 0)
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const double v = warp_sum_d(lane < kClusterWarps ? s_warp[lane][k] : 0.0);
            if (lane == 0) store_to_rank(&s_all[rank][k], 0, v);
        }
    cluster_sync();
    if (rank == 0 && warp == 0) {
#pragma unroll
        for (int k = 0; k < NS; ++k) acc[k] = warp_sum_d(lane < ranks ? s_all[lane][k] : 0.0);
        if (lane == 0) op.finish(acc, count);
    }
    if (*(volatile int*)&gave_up) {                      // give copies still in flight time to land
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }
    }
}

// A part of a device may have no room for the largest cluster.  Asked once per device.
cudaError_t terms_cluster_fits(bool* fits)
{
    static std::atomic<int> known[kDeviceSlots];         // 1: it fits, 2: it does not
    std::atomic<int>& k = known[device_slot()];
    if (!k.load(std::memory_order_acquire)) {
        static OncePerDevice allowed;
        cudaError_t e = allow_shared(terms_cluster_kernel, allowed);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(terms_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kClusterMost); cfg.blockDim = dim3(kClusterThreads); cfg.dynamicSmemBytes = (size_t)kClusterHolds * 24;
        cudaLaunchAttribute size;
        size.id = cudaLaunchAttributeClusterDimension;
        size.val.clusterDim.x = kClusterMost; size.val.clusterDim.y = size.val.clusterDim.z = 1;
        cfg.attrs = &size; cfg.numAttrs = 1;
        int clusters = 0;
        e = cudaOccupancyMaxActiveClusters(&clusters, terms_cluster_kernel, &cfg);
        if (e != cudaSuccess && e != cudaErrorInvalidClusterSize && e != cudaErrorLaunchOutOfResources) return e;
        if (e != cudaSuccess) cudaGetLastError();
        k.store(e == cudaSuccess && clusters > 0 ? 1 : 2, std::memory_order_release);
    }
    *fits = k.load(std::memory_order_acquire) == 1;
    return cudaSuccess;
}

// lost: without the copies, as if none of them landed (self-test).
cudaError_t launch_terms_cluster(const PpoOp<false>& op, int count, cudaStream_t s, bool lost = false)
{
    int ranks = 1;
    while (ranks < kClusterMost && ranks * kClusterEach < count) ranks *= 2;
    const int per_block = ((count + ranks - 1) / ranks + 3) / 4 * 4;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ranks); cfg.blockDim = dim3(kClusterThreads); cfg.dynamicSmemBytes = (size_t)per_block * 24; cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ranks; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, terms_cluster_kernel, op, count, per_block, lost);
}

}  // namespace
}  // namespace hts

extern "C" hts_status hts_a2c_terms(const float* logp, const float* values, const float* entropy, const float* returns,
                                    int64_t count, float* out3, void* cuda_stream)
{
    using namespace hts;
    if (!logp || !values || !entropy || !returns || !out3 || count < 1) return HTS_ERR_INVALID_ARG;
    const A2cOp op{logp, values, entropy, returns, out3, all_aligned16({logp, values, entropy, returns})};
    return launch_sums(op, (long long)count, static_cast<cudaStream_t>(cuda_stream));
}

namespace hts {
namespace {

enum class TermsForm { ByCount, TwoLaunches, ClusterLost };

hts_status ppo_terms(const float* logp_new, const float* logp_old, const float* values, const float* entropy, const float* advantages,
                     const float* returns, int64_t count, float clip, int32_t normalize_advantages, float* out4, void* cuda_stream, TermsForm form)
{
    if (!logp_new || !logp_old || !values || !entropy || !advantages || !returns || !out4 || count < 1) return HTS_ERR_INVALID_ARG;
    if (!(clip > 0.f) || std::isinf(clip)) return HTS_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const bool vec = all_aligned16({logp_new, logp_old, values, entropy, advantages, returns});
    const PpoOp<false> op{logp_new, logp_old, values, entropy, advantages, returns, out4, (double)clip, normalize_advantages != 0, vec};
    if (!normalize_advantages) return launch_sums(op, (long long)count, s);
    if (vec && count <= kClusterMost * kClusterHolds && form != TermsForm::TwoLaunches) {
        bool fits = false;
        HTS_CUDA(terms_cluster_fits(&fits));
        if (fits) {
            const cudaError_t e = launch_terms_cluster(op, (int)count, s, form == TermsForm::ClusterLost);
            if (e == cudaSuccess) { note_launch(); return HTS_OK; }
            // the current context may hold less of the device than the one that was asked
            if (e != cudaErrorInvalidClusterSize && e != cudaErrorLaunchOutOfResources) return cuda_fail(e, "terms_cluster_kernel");
            cudaGetLastError();
        }
    }
    const hts_status st = launch_sums(AdvStatsOp{advantages, all_aligned16({advantages})}, (long long)count, s);
    if (st != HTS_OK) return st;
    const SumsGrid grid = sums_grid((long long)count);
    if (grid.blocks <= 2LL * device_sm_count(device_slot()) && grid.per_block <= kThreads * kPerThread)
        return launch_sums<Form::EarlyTwo>(op, (long long)count, s);
    return launch_sums<Form::EarlyThree>(PpoOp<true>{logp_new, logp_old, values, entropy, advantages, returns, out4, (double)clip, true, vec},
                                         (long long)count, s);
}

}  // namespace
}  // namespace hts

extern "C" hts_status hts_ppo_terms(const float* logp_new, const float* logp_old, const float* values, const float* entropy,
                                    const float* advantages, const float* returns, int64_t count, float clip,
                                    int32_t normalize_advantages, float* out4, void* cuda_stream)
{
    return hts::ppo_terms(logp_new, logp_old, values, entropy, advantages, returns, count, clip, normalize_advantages, out4, cuda_stream,
                          hts::TermsForm::ByCount);
}

// For tests, not declared in hts.h.  The standardised means by two launches, as where the cluster does not fit, or (`lost`) by the
// cluster without its copies.
extern "C" hts_status hts_ppo_terms_selftest(const float* logp_new, const float* logp_old, const float* values, const float* entropy,
                                             const float* advantages, const float* returns, int64_t count, float clip, int32_t lost, float* out4,
                                             void* cuda_stream)
{
    return hts::ppo_terms(logp_new, logp_old, values, entropy, advantages, returns, count, clip, 1, out4, cuda_stream,
                          lost ? hts::TermsForm::ClusterLost : hts::TermsForm::TwoLaunches);
}

// ---- the learner's parameter update (Section 4.1 "Delayed gradient", Eq. 5) ---------------------------------
// theta_{j+1} = theta_j + eta * d with the gradient taken (by the caller) at theta_{j-1}.  With the RMSProp
// scaling of the hyper-parameter tables (momentum 0): v <- alpha v + (1 - alpha) g^2, d = g / (sqrt(v) + eps);
// without it d = g.  Elementwise and HBM-bound: 20 bytes per parameter, 22 with the bf16 copy that the actor's
// hts_policy_load_weights takes, written in the same pass.
namespace hts {
namespace {

template <bool PRECOND>
__device__ __forceinline__ float update_one(float theta, float g, float& v, float lr, float alpha, float eps)
{
    float d = g;
    if (PRECOND) {
        v = fmaf(alpha, v, (1.0f - alpha) * g * g);
        d = g / (sqrtf(v) + eps);
    }
    return fmaf(lr, d, theta);
}

// Four parameters per thread and pass when every array is 16-byte aligned (8 for the bf16 copy).
template <bool PRECOND, bool VEC>
__global__ void __launch_bounds__(256)
delayed_update_kernel(float* __restrict__ theta, const float* __restrict__ grad, float* __restrict__ sq_avg,
                      long long count, float lr, float alpha, float eps, __nv_bfloat16* __restrict__ theta_bf16)
{
    pdl_wait();
    pdl_trigger();
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long done = 0;
    if (VEC) {
        const long long quads = count >> 2;
        for (long long q = tid; q < quads; q += stride) {
            const float4 g = reinterpret_cast<const float4*>(grad)[q];
            float4 t = reinterpret_cast<float4*>(theta)[q];
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (PRECOND) v = reinterpret_cast<float4*>(sq_avg)[q];
            t.x = update_one<PRECOND>(t.x, g.x, v.x, lr, alpha, eps); t.y = update_one<PRECOND>(t.y, g.y, v.y, lr, alpha, eps);
            t.z = update_one<PRECOND>(t.z, g.z, v.z, lr, alpha, eps); t.w = update_one<PRECOND>(t.w, g.w, v.w, lr, alpha, eps);
            reinterpret_cast<float4*>(theta)[q] = t;
            if (PRECOND) reinterpret_cast<float4*>(sq_avg)[q] = v;
            if (theta_bf16) {
                __nv_bfloat162 lo = __floats2bfloat162_rn(t.x, t.y), hi = __floats2bfloat162_rn(t.z, t.w);
                reinterpret_cast<uint2*>(theta_bf16)[q] = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
            }
        }
        done = quads << 2;
    }
    for (long long i = done + tid; i < count; i += stride) {
        float v = PRECOND ? sq_avg[i] : 0.f;
        const float t = update_one<PRECOND>(theta[i], grad[i], v, lr, alpha, eps);
        theta[i] = t;
        if (PRECOND) sq_avg[i] = v;
        if (theta_bf16) theta_bf16[i] = __float2bfloat16_rn(t);
    }
}

}  // namespace
}  // namespace hts

extern "C" hts_status hts_delayed_update(float* theta, const float* grad, float* sq_avg_or_null, int64_t count,
                                         float lr, float alpha, float eps, void* theta_bf16_or_null, void* cuda_stream)
{
    using namespace hts;
    if (!theta || !grad || count < 1) return HTS_ERR_INVALID_ARG;
    if (!(lr == lr) || std::isinf(lr)) return HTS_ERR_INVALID_ARG;
    if (sq_avg_or_null && (!(alpha >= 0.f && alpha <= 1.f) || !(eps > 0.f) || std::isinf(eps))) return HTS_ERR_INVALID_ARG;
    long long blocks = (count + 256 * 4 - 1) / (256 * 4);
    const long long cap = 16LL * device_sm_count(device_slot());
    if (blocks > cap) blocks = cap;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    __nv_bfloat16* tb = static_cast<__nv_bfloat16*>(theta_bf16_or_null);
    const bool vec = (((uintptr_t)theta | (uintptr_t)grad | (uintptr_t)sq_avg_or_null) & 15u) == 0 && ((uintptr_t)tb & 7u) == 0;
    const unsigned gb = (unsigned)blocks;
    const long long n = (long long)count;
    auto kernel = sq_avg_or_null ? (vec ? delayed_update_kernel<true, true> : delayed_update_kernel<true, false>)
                                 : (vec ? delayed_update_kernel<false, true> : delayed_update_kernel<false, false>);
    HTS_CUDA(launch_pdl(kernel, dim3(gb), dim3(256), 0, s, theta, grad, sq_avg_or_null, n, lr, alpha, eps, tb));
    note_launch();
    return HTS_OK;
}
