// Tensor-core path of the actor step (bf16 weights): the convolution and FC layers of the
// policy-value network (Appendix F.1 / F.2) as tcgen05 GEMMs with TMA-fed shared-memory
// operands and fp32 accumulators in tensor memory.
//
// Formulation.  Activations live in HBM/L2 as row-major [pixel rows, channels] matrices.
// A k x k / s convolution with k = 2s is a 2x2/1 convolution on the space-to-depth(s) image,
// and a stride-1 convolution on a flat pixel grid is a sum over taps of row-shifted GEMMs:
//     D[m, o] = sum_tap sum_c X[m + dy*W_in + dx, c] * W[o, tap, c]
// computed for whole grid rows (conv_res_tc.cu); columns whose x falls outside the output extent are discarded by the epilogue.
// The FC layer is a GEMM with a fixed split of K into ranges, whose sums are added in index order here, in fc_tc.cu or by
// the heads kernel, so nothing depends on the batch size.
//
// Operand type.  Both MMA operands are fp16 (kind::f16, fp32 accumulation).  The caller's bf16
// weights are multiplied by a per-layer power of two that brings the largest magnitude just
// below 2^15 and converted to fp16: exact for every weight within 2^-29 of the largest (bf16
// has 8 significant bits, fp16 has 11); the epilogue divides the power of two out again.
// Activations are stored as fp16 (clamped at the largest finite value): 11 significant bits
// instead of bf16's 8, which keeps the logits well inside the 2e-2 parity bound.
#include <new>
#include <type_traits>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include "common.cuh"
#include "tc_ptx.cuh"
#include "tc_host.cuh"
#include "conv1_tc.cuh"
#include "conv_res_tc.cuh"
#include "fc_tc.cuh"
#include "conv_stack_tc.cuh"

namespace hts {
using namespace tc;

namespace {

constexpr int BM = 128;                 // rows per tile = TMEM lanes
constexpr int BK = 64;                  // 16-bit elements per K chunk = one 128-byte swizzle row
constexpr int A_BYTES = BM * BK * 2;    // 16 KiB
enum { L_CONV1 = 0, L_CONV2, L_CONV3, L_FC, L_COUNT };

// ---- FC for small batches with the weights resident: one CTA per (column tile, K range, row tile).
// A CTA asks for its whole weight slice (nk chunks of 128 x 64) before it waits for the previous kernel; a CTA of
// this kernel cannot start before the previous kernel's CTA has left its SM, but the hand-over from the last of
// those to the release of the wait (about 1.4 us) is enough for most of the slice.  After the wait only
// activations cross the SM's L2 port: 112 KB per row tile instead of 224 KB.  Used while every CTA has one row
// tile (n <= 640 for 4 x 84 x 84 frames: 31.0 us per step at n = 256, 31.5 with weights and activations copied together);
// from there on pairs of SMs (fc_tc.cu) are faster.  K ranges, the order inside them and the partial planes are the same
// there: the same bits.
constexpr int FCB_STAGES = 5;                   // activation chunks in flight (16 KiB each)
constexpr int FCB_MAX_NK = 7;                   // weight chunks a CTA can keep: 7 x 16 KiB
constexpr int FCB_STAGE_FLOATS = 4 * 32 * 36;   // the epilogue warps' transposing buffers

struct FcbParams {
    int nk;                             // K chunks of one range
    int n_env;                          // valid rows
    int row0;                           // the first one's row of the activations
    const float* inv_scale;
    float* out_f32;                     // partial planes [range][rows][512]
    size_t split_stride;
    int* status;
};

__global__ void __launch_bounds__(192)
fc_resident_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const FcbParams p)
{
    constexpr int BN = 128;
    constexpr int B_BYTES = BN * BK * 2;
    extern __shared__ uint8_t smem_raw[];
    constexpr int kBars = FCB_MAX_NK + 2 * FCB_STAGES + 1;
    __shared__ uint64_t bars[kBars];
    uint64_t *b_full = bars, *a_full = bars + FCB_MAX_NK, *a_empty = a_full + FCB_STAGES, *acc_full = a_empty + FCB_STAGES;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
    uint8_t* sm_a = sm + FCB_MAX_NK * B_BYTES;
    const uint32_t a_base = base + FCB_MAX_NK * B_BYTES;
    float* sm_stage = reinterpret_cast<float*>(sm_a + FCB_STAGES * A_BYTES);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * BN, range = blockIdx.y, m0 = blockIdx.z * BM;
    volatile int* abortp = &abort_flag;

    if (warp == 0) {
        static_assert(kBars <= 32, "a lane initialises one barrier");
        if (lane < kBars) mbar_init(&bars[lane], 1);
        fence_barrier_init();
        __syncwarp();
        if (lane == 0) {                                 // the weights do not depend on the previous kernel
            for (int kc = 0; kc < p.nk; ++kc) {
                mbar_arrive_expect_tx(&b_full[kc], B_BYTES);
                tma_load_2d(sm + kc * B_BYTES, &tmB, (range * p.nk + kc) * BK, n0, &b_full[kc]);
            }
        }
    } else if (warp == 1) {
        tmem_alloc(&tmem_base_slot, BN);
    } else if (warp == 2 && lane == 0) {
        abort_flag = 0;
        tma_prefetch_desc(&tmA);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_d = tmem_base_slot;
    pdl_wait();
    pdl_trigger();

    if (warp == 0) {
        if (lane == 0) {
            for (int kc = 0; kc < p.nk; ++kc) {
                const int s = kc % FCB_STAGES;
                if (!mbar_wait(&a_empty[s], (((uint32_t)(kc / FCB_STAGES)) & 1u) ^ 1u, abortp, p.status, 71)) break;
                mbar_arrive_expect_tx(&a_full[s], A_BYTES);
                tma_load_2d(sm_a + s * A_BYTES, &tmA, (range * p.nk + kc) * BK, p.row0 + m0, &a_full[s]);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = instr_desc_f16(0, BM, BN);
            bool alive = true;
            for (int kc = 0; kc < p.nk; ++kc) {
                const int s = kc % FCB_STAGES;
                if (!mbar_wait(&b_full[kc], 0, abortp, p.status, 72)) { alive = false; break; }
                if (!mbar_wait(&a_full[s], ((uint32_t)(kc / FCB_STAGES)) & 1u, abortp, p.status, 73)) { alive = false; break; }
                tc_fence_after();
                const uint64_t adesc = smem_desc_sw128(a_base + s * A_BYTES);
                const uint64_t bdesc = smem_desc_sw128(base + kc * B_BYTES);
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                    mma_f16_ss(tmem_d, adesc + 2 * k, bdesc + 2 * k, idesc, (kc | k) != 0);
                mma_commit(&a_empty[s]);
            }
            if (alive) mma_commit(acc_full);
        }
    } else {
        // epilogue warps 2..5: warp w may touch TMEM lanes [32*(w%4), 32*(w%4)+32)
        const int q = warp & 3;
        const float inv = *p.inv_scale;
        float* stage = sm_stage + (warp - 2) * (32 * 36);
        const int rl = lane >> 3, c4 = (lane & 7) * 4;
        if (mbar_wait_warp(acc_full, 0, abortp, p.status, 74)) {
            tc_fence_after();
            // one row per thread arrives; each warp turns its 32 x 32 blocks through shared memory so that eight
            // lanes write one full 128-byte line
            float* dst = p.out_f32 + range * p.split_stride + (size_t)(m0 + q * 32) * 512 + n0;
#pragma unroll
            for (int c = 0; c < BN; c += 32) {
                uint32_t v[32];
                tmem_ld_32x32(tmem_d + ((uint32_t)(q * 32) << 16) + c, v);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    *reinterpret_cast<float4*>(stage + lane * 36 + j) =
                        make_float4(__uint_as_float(v[j]) * inv, __uint_as_float(v[j + 1]) * inv,
                                    __uint_as_float(v[j + 2]) * inv, __uint_as_float(v[j + 3]) * inv);
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rr = 4 * i + rl;
                    const float4 val = *reinterpret_cast<const float4*>(stage + rr * 36 + c4);
                    if (m0 + q * 32 + rr < p.n_env) *reinterpret_cast<float4*>(dst + (size_t)rr * 512 + c + c4) = val;
                }
                __syncwarp();
            }
        }
    }
    if (*abortp) {                                      // give copies still in flight time to land
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_d, BN);
}

// ---- weight scaling and packing ---------------------------------------------------------------
// Two launches: the largest magnitude of each layer (the last block to finish turns them into scales), then every
// layer scaled, converted and laid out.  They follow each parameter update, so launches count: 18 separate ones took
// 125 us (47 of them in a 64-block pass over the dense layer); two are 14, and 9.4 since the second reads its rows while
// the first runs.
struct LoadTcParams {
    const __nv_bfloat16* w[L_COUNT];    // conv1, conv2, conv3, dense
    int n[L_COUNT];
    unsigned* absmax;                   // [L_COUNT], then the ticket; zero between calls
    float *scale, *inv_scale;
    float conv1_extra;
    int C, P3;
    __half* wp[L_COUNT];
    const __nv_bfloat16* f[8];          // biases and heads: kept as fp32
    float* fdst[8];
    int fn[8];
};
constexpr int kAbsmaxPerSm = 4;         // blocks of the first

__global__ void __launch_bounds__(256) absmax_kernel(const LoadTcParams p)
{
    __shared__ bool s_last;
    __shared__ unsigned s_max[8][L_COUNT];
    const int tid = blockIdx.x * 256 + threadIdx.x, threads = gridDim.x * 256;
    pdl_wait();
    pdl_trigger();
#pragma unroll
    for (int l = 0; l < L_COUNT; ++l) {
        unsigned m = 0;                                 // finite magnitudes order like their bits
        auto take = [&](uint32_t bits) { bits &= 0x7fffu; if (bits < 0x7f80u) m = max(m, bits); };
        int done = 0;
        if (((uintptr_t)p.w[l] & 15) == 0) {
            const uint4* v = reinterpret_cast<const uint4*>(p.w[l]);
            for (int i = tid; i < p.n[l] / 8; i += threads) {
                const uint4 q = v[i];
                take(q.x); take(q.x >> 16); take(q.y); take(q.y >> 16); take(q.z); take(q.z >> 16); take(q.w); take(q.w >> 16);
            }
            done = p.n[l] / 8 * 8;
        }
        for (int i = done + tid; i < p.n[l]; i += threads) take(reinterpret_cast<const uint16_t*>(p.w[l])[i]);
        m = __reduce_max_sync(0xffffffffu, m);
        if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5][l] = m;
    }
    __syncthreads();
    if (threadIdx.x < L_COUNT) {                        // one atomic per block and layer: they all meet at one address
        unsigned m = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) m = max(m, s_max[w][threadIdx.x]);
        if (m) atomicMax(p.absmax + threadIdx.x, m << 16);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(p.absmax + L_COUNT, 1u) == gridDim.x - 1;
    __syncthreads();
    if (s_last && threadIdx.x <= L_COUNT) {
        const int l = threadIdx.x;
        __threadfence();
        const float mx = __uint_as_float(atomicExch(p.absmax + l, 0u));      // and ready for the next call
        if (l == L_COUNT) return;
        // scale = 2^(14 - floor(log2 max)): the largest weight lands in [2^14, 2^15)
        int e = 0;
        float s = 1.f;
        if (mx > 0.f) { frexpf(mx, &e); s = ldexpf(1.f, 15 - e); }        // mx = f * 2^e, f in [0.5, 1)
        p.scale[l] = s;
        p.inv_scale[l] = (l == L_CONV1 ? p.conv1_extra : 1.f) / s;
    }
}
__device__ __forceinline__ __half scaled_h(__nv_bfloat16 w, float s) { return __float2half_rn(__bfloat162float(w) * s); }

//   conv1: row dy*64 + dx*32 + o, column c*16 + uy*4 + ux       value w1[o][c][4dy+uy][4dx+ux]
//   conv2: [o][(tap*2 + half)*64 + j], c' = half*64 + j = (uy*2+ux)*32 + c, tap = dy*2+dx, value w2[o][c][2dy+uy][2dx+ux]
//   conv3: [o][(dy*3+dx)*64 + c]                                value w3[o][c][dy][dx]
//   dense: [o][pix*64 + c] (activations are stored pixel-major)  value wfc[o][c*P3 + pix]
// Blocks 0..511 take one row of the dense layer each and turn it through shared memory (rows of up to 16384 columns;
// wider ones are read with a stride); the rest one element per thread.
constexpr int kPackRow = 16384;
__global__ void __launch_bounds__(256) pack_kernel(const LoadTcParams p)
{
    __shared__ __nv_bfloat16 s_row[kPackRow];
    if (blockIdx.x < 512) {
        const int o = blockIdx.x, F = 64 * p.P3;
        const __nv_bfloat16* src = p.w[L_FC] + (size_t)o * F;
        if (F <= kPackRow) {                            // the caller's weights are older than the pass over them
            for (int i = threadIdx.x; i < F; i += 256) s_row[i] = src[i];
            __syncthreads();
            src = s_row;
        }
        pdl_wait();
        const float s = p.scale[L_FC];
        __half* dst = p.wp[L_FC] + (size_t)o * F;
        for (int k = threadIdx.x; k < F; k += 256) dst[k] = scaled_h(src[(k & 63) * p.P3 + (k >> 6)], s);
        return;
    }
    pdl_wait();
    int i = (blockIdx.x - 512) * 256 + threadIdx.x;
    const int K = 16 * p.C;
    if (i < 128 * K) {
        const int row = i / K, k = i - row * K, dy = row >> 6, dx = (row >> 5) & 1, o = row & 31;
        const int c = k >> 4, uy = (k >> 2) & 3, ux = k & 3;
        p.wp[L_CONV1][i] = scaled_h(p.w[L_CONV1][((o * p.C + c) * 8 + (4 * dy + uy)) * 8 + (4 * dx + ux)], p.scale[L_CONV1]);
        return;
    }
    i -= 128 * K;
    if (i < 64 * 512) {
        const int o = i / 512, k = i % 512, tap = k / 128, cp = k % 128;
        const int dy = tap >> 1, dx = tap & 1, uy = (cp / 32) >> 1, ux = (cp / 32) & 1, c = cp % 32;
        p.wp[L_CONV2][i] = scaled_h(p.w[L_CONV2][((o * 32 + c) * 4 + (2 * dy + uy)) * 4 + (2 * dx + ux)], p.scale[L_CONV2]);
        return;
    }
    i -= 64 * 512;
    if (i < 64 * 576) {
        const int o = i / 576, k = i % 576, tap = k / 64, c = k % 64;
        p.wp[L_CONV3][i] = scaled_h(p.w[L_CONV3][(o * 64 + c) * 9 + tap], p.scale[L_CONV3]);
        return;
    }
    i -= 64 * 576;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (i < p.fn[k]) {
            p.fdst[k][i] = __bfloat162float(p.f[k][i]);
            return;
        }
        i -= p.fn[k];
    }
}

// ---- parity taps: internal layouts -> fp32 NCHW ----------------------------------------------------
// Rows of conv1's output (s2d) and conv2's are ordered (y, env, x), `W_rows` to an environment and grid row and env_rows
// environments to a grid row; conv3's (env, y, x).
enum { TAP_S2D, TAP_ROWS, TAP_PIXELS };
__global__ void tap_rows_kernel(const __half* __restrict__ src, float* __restrict__ dst, int n, int Cc,
                                int Ho, int Wo, int form, size_t env_rows, int W_rows)
{
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t total = (size_t)n * Cc * Ho * Wo;
    if (idx >= total) return;
    const int x = (int)(idx % Wo), y = (int)((idx / Wo) % Ho), c = (int)((idx / ((size_t)Wo * Ho)) % Cc);
    const size_t e = idx / ((size_t)Wo * Ho * Cc);
    size_t off;
    if (form == TAP_S2D) off = (((size_t)(y >> 1) * env_rows + e) * W_rows + (x >> 1)) * (4 * Cc) + ((y & 1) * 2 + (x & 1)) * Cc + c;
    else if (form == TAP_ROWS) off = (((size_t)y * env_rows + e) * W_rows + x) * Cc + c;
    else off = ((e * Ho + y) * Wo + x) * Cc + c;
    dst[idx] = __half2float(src[off]);
}

inline unsigned nblk(size_t total, int th) { return (unsigned)((total + th - 1) / th); }

hts_status launch_fc_resident(const CUtensorMap& a, const CUtensorMap& b, const FcbParams& p, int ranges, int m_tiles,
                              cudaStream_t s)
{
    constexpr int smem = FCB_MAX_NK * 128 * BK * 2 + FCB_STAGES * A_BYTES + FCB_STAGE_FLOATS * 4 + 1024;
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(fc_resident_kernel, allowed));
    HTS_CUDA(launch_pdl(fc_resident_kernel, dim3(4, ranges, m_tiles), dim3(192), (size_t)smem, s, a, b, p));
    note_launch();
    return HTS_OK;
}

}  // namespace

struct TcState {
    Geometry g;
    int max_batch;
    int H1s, W1s, P1s;          // space-to-depth(2) grid of the conv1 output
    int P2, P3;
    int splits, cps;            // FC split-K
    bool fresh = false;         // no step has been enqueued since the weights were packed
    unsigned long long fresh_capture = 0;   // the stream capture that packing belongs to, 0 = none
    bool h_final = false;       // the last forward pass wrote the finished hidden layer, not planes to be added up
    int planes = 0;             // how many of those
    // packed weights
    Conv1Plan pl1;
    Conv1MapCache maps1;
    __half *w1p, *w2p, *w3p, *wfcp;
    float *b1, *b2, *b3, *bfc, *whead, *bhead;
    unsigned* absmax;           // [L_COUNT] and a ticket, zero between calls
    float *scale, *inv_scale;   // [L_COUNT] each
    // workspace
    __half *a1s, *a2, *a3;
    float *hpart, *h;
    CUtensorMap mW1, mA2, mB2, mA3, mB3, mAfc, mBfc, mBfcPair, mT1, mT2;
    bool stacked;               // the frames fit the kernel that runs all three convolutions
    ConvStackParams stack;
    int* status;
};

hts_status tc_check_geometry(const Geometry& g)
{
    Conv1Plan pl;
    if (!conv1_plan(g, &pl)) return HTS_ERR_SHAPE;
    if (g.F % BK) return HTS_ERR_SHAPE;
    // the frames this path has been made for: conv2's input grid at most 31 wide (frames of 252 columns) and of 2048 pixels
    if (pl.P1s > 2048 || pl.W1s > 31) return HTS_ERR_SHAPE;
    return HTS_OK;
}

hts_status tc_create(const Geometry& g, int max_batch, int* status, TcState** out,
                     bool (*alloc)(void* ctx, void** p, size_t bytes), void* alloc_ctx)
{
    TcState* t = new (std::nothrow) TcState();
    if (!t) return HTS_ERR_ALLOC;
    t->g = g; t->max_batch = max_batch; t->status = status;
    if (tc_check_geometry(g) != HTS_OK || !conv1_plan(g, &t->pl1)) { delete t; return HTS_ERR_SHAPE; }
    t->H1s = t->pl1.H1s; t->W1s = t->pl1.W1s; t->P1s = t->pl1.P1s;
    t->P2 = g.H2 * g.W2; t->P3 = g.H3 * g.W3;
    const int chunks = g.F / BK;
    t->splits = 1;
    for (int s = 8; s >= 1; --s) if (chunks % s == 0) { t->splits = s; break; }
    t->cps = chunks / t->splits;
    const size_t nb = (size_t)max_batch;
    // one allocation for all buffers: sizes first, then the pointers
    uint8_t* base = nullptr;
    for (int pass = 0; pass < 2; ++pass) {
        size_t total = 0;
        auto A = [&](auto** p, size_t count) {
            *p = reinterpret_cast<std::remove_reference_t<decltype(*p)>>(base + total);
            total += (count * sizeof(**p) + 256 + 1023) & ~(size_t)1023;
        };
        A(&t->w2p, (size_t)64 * 512); A(&t->w3p, (size_t)64 * 576); A(&t->wfcp, (size_t)512 * g.F);
        A(&t->w1p, (size_t)128 * 16 * g.C); A(&t->b1, 32); A(&t->b2, 64); A(&t->b3, 64); A(&t->bfc, 512);
        A(&t->whead, (size_t)(g.A + 1) * 512); A(&t->bhead, (size_t)g.A + 1);
        A(&t->absmax, L_COUNT + 1); A(&t->scale, L_COUNT); A(&t->inv_scale, L_COUNT);
        A(&t->a1s, nb * t->P1s * 128); A(&t->a2, nb * t->P2 * 64); A(&t->a3, nb * g.F);
        A(&t->hpart, (size_t)t->splits * nb * 512); A(&t->h, nb * 512);
        if (pass == 0 && !alloc(alloc_ctx, reinterpret_cast<void**>(&base), total)) { delete t; return HTS_ERR_ALLOC; }
    }
    // cells of an odd-sized s2d border that conv1 never writes must hold finite numbers
    if (cudaMemset(t->a1s, 0, nb * t->P1s * 128 * 2) != cudaSuccess) { delete t; return cuda_fail(cudaGetLastError(), "cudaMemset"); }
    if (cudaMemset(t->absmax, 0, (L_COUNT + 1) * sizeof(unsigned)) != cudaSuccess) { delete t; return cuda_fail(cudaGetLastError(), "cudaMemset"); }
    const bool ok = make_map(&t->mW1, t->w1p, 128, 16 * g.C, (uint64_t)32 * g.C, 64) &&
         make_map(&t->mA2, t->a1s, nb * t->P1s, 128, 256, kConvRowsBox<2>) && make_map(&t->mB2, t->w2p, 64, 512, 1024, 64) &&
         make_map(&t->mA3, t->a2, nb * t->P2, 64, 128, kConvRowsBox<3>) && make_map(&t->mB3, t->w3p, 64, 576, 1152, 64) &&
         make_map(&t->mAfc, t->a3, nb, g.F, (uint64_t)g.F * 2, BM) && make_map(&t->mBfc, t->wfcp, 512, g.F, (uint64_t)g.F * 2, 128) &&
         make_map(&t->mBfcPair, t->wfcp, 512, g.F, (uint64_t)g.F * 2, 64);
    if (!ok) { delete t; return HTS_ERR_CUDA; }
    t->stack = ConvStackParams{};
    t->stacked = conv_stack_plan(g, &t->stack);
    ConvStackParams& cs = t->stack;
    cs.b1 = t->b1; cs.b2 = t->b2; cs.b3 = t->b3; cs.inv1 = t->inv_scale + L_CONV1; cs.inv2 = t->inv_scale + L_CONV2; cs.inv3 = t->inv_scale + L_CONV3;
    cs.a3 = t->a3; cs.status = status;
    if (t->stacked && !(make_grid_map(&t->mT1, t->a1s, 128, t->W1s, nb, t->H1s) && make_grid_map(&t->mT2, t->a2, 64, g.W2, nb, g.H2))) { delete t; return HTS_ERR_CUDA; }
    *out = t;
    return HTS_OK;
}

void tc_destroy(TcState* t) { delete t; }

namespace {

unsigned long long capture_of(cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamGetCaptureInfo(s, &st, &id) != cudaSuccess) { cudaGetLastError(); return 0; }
    return st == cudaStreamCaptureStatusActive ? id : 0;
}

// May the first layer of a step start before its predecessor has ended?  Not where that can be the packing of the weights
// it loads.  A step recorded into a graph does not follow a packing that runs outside of it: the next one may.
bool first_layer_dependent(TcState* t, cudaStream_t s)
{
    if (!t->fresh) return true;
    const unsigned long long now = capture_of(s);
    if (now == 0 || now == t->fresh_capture) t->fresh = false;
    return false;
}

}  // namespace

hts_status tc_load_weights(TcState* t, const hts_weights& w, cudaStream_t s)
{
    const Geometry& g = t->g;
    auto bf = [](const void* p) { return static_cast<const __nv_bfloat16*>(p); };
    LoadTcParams p{};
    // conv1 feeds raw bytes as fp16 subnormals (b * 2^-24): its accumulator scale undoes that and the /255
    p.absmax = t->absmax; p.scale = t->scale; p.inv_scale = t->inv_scale; p.conv1_extra = 16777216.0f / 255.0f; p.C = g.C; p.P3 = t->P3;
    const void* ws[L_COUNT] = {w.conv1_w, w.conv2_w, w.conv3_w, w.fc_w};
    const int wn[L_COUNT] = {32 * g.C * 64, 64 * 512, 64 * 576, 512 * g.F};
    __half* wp[L_COUNT] = {t->w1p, t->w2p, t->w3p, t->wfcp};
    for (int l = 0; l < L_COUNT; ++l) { p.w[l] = bf(ws[l]); p.n[l] = wn[l]; p.wp[l] = wp[l]; }
    struct It { const void* p; float* q; int n; };
    const It items[8] = {{w.conv1_b, t->b1, 32}, {w.conv2_b, t->b2, 64},
                         {w.conv3_b, t->b3, 64}, {w.fc_b, t->bfc, 512}, {w.pi_w, t->whead, g.A * 512},
                         {w.v_w, t->whead + (size_t)g.A * 512, 512}, {w.pi_b, t->bhead, g.A}, {w.v_b, t->bhead + g.A, 1}};
    int rest = 128 * 16 * g.C + 64 * 512 + 64 * 576;
    for (int k = 0; k < 8; ++k) { p.f[k] = bf(items[k].p); p.fdst[k] = items[k].q; p.fn[k] = items[k].n; rest += items[k].n; }
    HTS_CUDA(launch_pdl(absmax_kernel, dim3(kAbsmaxPerSm * device_sm_count(device_slot())), dim3(256), 0, s, p));
    note_launch();
    HTS_CUDA(launch_pdl(pack_kernel, dim3(512 + nblk(rest, 256)), dim3(256), 0, s, p));
    note_launch();
    t->fresh = true;
    t->fresh_capture = capture_of(s);
    return HTS_OK;
}

hts_status tc_forward(TcState* t, const uint8_t* obs, const Indexing& ix, int n, Profiler& prof, cudaStream_t s)
{
    const Geometry& g = t->g;
    hts_status st;
    const bool dependent = first_layer_dependent(t, s);
    const size_t row0 = (size_t)ix.row0;
    if (t->stacked && n <= conv_stack_envs(t->stack) * device_sm_count(device_slot())) {
        ConvStackParams c = t->stack;
        c.obs = obs; c.slots = ix.slots; c.pool = ix.pool; c.n = n; c.row0 = ix.row0;
        prof.begin(K_CONV1, s);
        st = conv_stack_launch(t->mW1, t->mB2, t->mB3, t->mT1, t->mT2, c, dependent, s);
        if (st != HTS_OK) return st;
        prof.end(K_CONV1, s);
    } else {
        prof.begin(K_CONV1, s);
        st = conv1_launch(t->pl1, t->mW1, t->maps1, obs, ix, n, t->b1, t->inv_scale + L_CONV1, t->a1s + row0 * t->W1s * 128, t->max_batch, t->status, dependent, s);
        if (st != HTS_OK) return st;
        prof.end(K_CONV1, s);

        // conv2: 2x2 taps on the s2d grid [H1s, W1s] with 128 channels -> [H2, W2] x 64, rows (y, env, x) again
        const size_t nb = (size_t)t->max_batch;
        ConvRowsParams c{};
        c.status = t->status; c.n_env = n;
        c.W_in = t->W1s; c.H_out = g.H2; c.W_out = g.W2; c.in_plane = (int)(nb * t->W1s); c.col0 = ix.row0 * t->W1s;
        c.tiles = (int)nblk((size_t)n * c.W_in, BM);
        c.bias = t->b2; c.inv_scale = t->inv_scale + L_CONV2;
        c.out_env = (size_t)g.W2 * 64; c.out_y = nb * g.W2 * 64; c.out = t->a2 + row0 * c.out_env;
        prof.begin(K_CONV2, s);
        st = conv_rows_launch<2, 2, 2>(t->mA2, t->mB2, c, s);
        if (st != HTS_OK) return st;
        prof.end(K_CONV2, s);
        // conv3: 3x3 taps on [H2, W2] x 64 -> [H3, W3] x 64, an environment's pixels together: a row of the dense layer's input
        c.W_in = g.W2; c.H_out = g.H3; c.W_out = g.W3; c.in_plane = (int)(nb * g.W2); c.col0 = ix.row0 * g.W2;
        c.tiles = (int)nblk((size_t)n * c.W_in, BM);
        c.bias = t->b3; c.inv_scale = t->inv_scale + L_CONV3;
        c.out_env = (size_t)g.F; c.out_y = (size_t)g.W3 * 64; c.out = t->a3 + row0 * c.out_env;
        prof.begin(K_CONV3, s);
        st = conv_rows_launch<3, 3, 1>(t->mA3, t->mB3, c, s);
        if (st != HTS_OK) return st;
        prof.end(K_CONV3, s);
    }
    // FC: [n, F] x [512, F]^T, K split into ranges.  Weights resident per CTA when a range is at most seven chunks and every
    // CTA gets one row tile, pairs of SMs otherwise.
    prof.begin(K_FC, s);
    const int m_tiles = (int)nblk(n, BM);
    if (t->cps <= FCB_MAX_NK && m_tiles <= device_sm_count(device_slot()) / (4 * t->splits)) {
        const FcbParams fp{t->cps, n, ix.row0, t->inv_scale + L_FC, t->hpart + row0 * 512, (size_t)t->max_batch * 512, t->status};
        t->planes = t->splits;
        t->h_final = false;
        st = launch_fc_resident(t->mAfc, t->mBfc, fp, t->splits, m_tiles, s);
    } else {
        const FcPairPlan plan = fc_pair_plan(n, t->splits);
        const FcPairParams fp{t->splits, t->cps, plan.group, n, ix.row0, t->bfc, t->inv_scale + L_FC, t->h + row0 * 512, t->hpart + row0 * 512, (size_t)t->max_batch * 512, t->status};
        t->planes = plan.planes;
        t->h_final = plan.planes == 1;
        st = fc_pair_launch(t->mAfc, t->mBfcPair, fp, plan.wide, s);
    }
    if (st != HTS_OK) return st;
    prof.end(K_FC, s);
    return HTS_OK;
}

hts_status tc_heads(TcState* t, const int32_t* env_ids, const int32_t* t_per_env, int32_t tt, uint64_t seed, int n,
                    const Indexing& ix, int32_t* actions, float* logp, float* values, float* entropy, float* logits,
                    cudaStream_t s, const int32_t* given_actions)
{
    float *h = t->h + (size_t)ix.row0 * 512, *planes = t->hpart + (size_t)ix.row0 * 512;
    if (t->h_final)        // the FC kernel wrote relu(bias + sum of the K ranges) itself
        return launch_heads(h, 1, 0, nullptr, t->whead, t->bhead, t->g.A, env_ids, t_per_env, tt, seed, n, ix, t->status,
                            actions, logp, values, entropy, logits, nullptr, s, given_actions);
    return launch_heads(planes, t->planes, (size_t)t->max_batch * 512, t->bfc, t->whead, t->bhead, t->g.A, env_ids,
                        t_per_env, tt, seed, n, ix, t->status, actions, logp, values, entropy, logits, h, s, given_actions);
}

hts_status tc_read_activation(TcState* t, int layer, int n, float* out, cudaStream_t s)
{
    const Geometry& g = t->g;
    if (layer == 4) {
        HTS_CUDA(cudaMemcpyAsync(out, t->h, (size_t)n * 512 * sizeof(float), cudaMemcpyDeviceToDevice, s));
        return HTS_OK;
    }
    if (layer == 1)
        tap_rows_kernel<<<nblk((size_t)n * 32 * g.H1 * g.W1, 256), 256, 0, s>>>(t->a1s, out, n, 32, g.H1, g.W1, TAP_S2D, t->max_batch, t->W1s);
    else if (layer == 2)
        tap_rows_kernel<<<nblk((size_t)n * 64 * g.H2 * g.W2, 256), 256, 0, s>>>(t->a2, out, n, 64, g.H2, g.W2, TAP_ROWS, t->max_batch, g.W2);
    else
        tap_rows_kernel<<<nblk((size_t)n * 64 * g.H3 * g.W3, 256), 256, 0, s>>>(t->a3, out, n, 64, g.H3, g.W3, TAP_PIXELS, 0, 0);
    HTS_LAUNCH_CHECK("tap_rows_kernel");
    return HTS_OK;
}

}  // namespace hts
