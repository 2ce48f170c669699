// Gradient of the learner objective with respect to the twelve parameter tensors: the quantity Eq. 4 of
// the paper estimates and Eq. 5 adds to the parameters,
//
//     J-hat = (1/n) sum_i [ S_i - value_coef (R_i - V(s_i))^2 + entropy_coef H(pi(.|s_i)) ],
//
// S_i = log pi(a_i|s_i) A_i (actor-critic; the advantage is data) or the clipped surrogate
// min(rho_i A_i, clip(rho_i, 1-clip, 1+clip) A_i), rho_i = exp(log pi(a_i|s_i) - logp_old_i) (PPO).
//
// The forward pass is that of the fp32 actor step: a ReLU passes the gradient exactly where the step's output is
// positive.  The data and weight gradients of the four hidden layers run on the tensor cores at fp32 accuracy
// (x3_gemm.cuh); the two heads, less than half a percent of the work, are fp32 CUDA-core kernels.
// Every sum runs in an order fixed by the batch size (no atomics): a weight gradient is summed per range of rows and
// the ranges are then added in index order.
#include <new>
#include "common.cuh"
#include "x3_gemm.cuh"

namespace hts {
namespace {

typedef __nv_bfloat16 bf16;

// ---- frames as the first convolution's operand -----------------------------------------------------------------
// uint8 [n,C,H,W] -> bf16 [n * (H/4)(W/4)][16 Cp], column c*16 + uy*4 + ux = x[c][4Y+uy][4X+ux] (a byte is exact);
// Cp = C rounded up to a multiple of 4, the added channels are zero.
// Bound by memory (87 MB for 1024 frames of 84 x 84 x 4, 18 us), where conv1 is bound by its multiply-adds.  Where conv1 has blocks
// of 32 strips for more than three to an SM, this runs beside its last ones: it begins when they have all begun (its inputs are
// ready then) and waits for them with its last block only, so that its own end means theirs.  Gradient without the forward pass, us,
// before conv1 / beside it: 160 of 84 x 84 x 4 99.1 / 96.5, 1024 316 / 312, 512 of 72 x 96 x 16 238 / 221; where all of conv1's blocks are on
// the device at once the two crowd each other: 80 of 84 x 84 x 4 71.5 / 83.5, 40 of 72 x 96 x 16 64 / 105.
struct FramesParams {
    const uint8_t* obs;
    int C, Cp, H, W;
    size_t items;                       // (position, channel), channel fastest
    bool words;                         // frames 4-byte aligned
    bf16* x0;
    bool beside;                        // launched behind conv1
};
__global__ void __launch_bounds__(256) frames_kernel(const FramesParams p)
{
    if (!p.beside || blockIdx.x == gridDim.x - 1) pdl_wait();
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= p.items) return;
    const int c = (int)(idx % p.Cp);
    const size_t pos = idx / p.Cp;
    const int W0 = p.W / 4, G0 = W0 * (p.H / 4);
    const size_t e = pos / G0;
    const int cell = (int)(pos - e * G0), Y = cell / W0, X = cell - Y * W0;
    uint32_t out[8];
#pragma unroll
    for (int uy = 0; uy < 4; ++uy) {
        uint32_t w = 0;
        if (c < p.C) {
            const uint8_t* src = p.obs + ((e * p.C + c) * p.H + 4 * Y + uy) * p.W + 4 * X;
            if (p.words) w = *reinterpret_cast<const uint32_t*>(src);
            else w = src[0] | (uint32_t)src[1] << 8 | (uint32_t)src[2] << 16 | (uint32_t)src[3] << 24;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float lo = (float)((w >> (16 * h)) & 0xffu), hi = (float)((w >> (16 * h + 8)) & 0xffu);
            out[2 * uy + h] = (__float_as_uint(lo) >> 16) | (__float_as_uint(hi) & 0xffff0000u);
        }
    }
    uint4* dst = reinterpret_cast<uint4*>(p.x0 + idx * 16);
    dst[0] = make_uint4(out[0], out[1], out[2], out[3]);
    dst[1] = make_uint4(out[4], out[5], out[6], out[7]);
}

// ---- fp32 weights as three bf16 planes in the layouts of the contractions ---------------------------------------
//   w2p [3][64][tap * 128 + (uy*2+ux)*32 + c]    value w2[o][c][2dy+uy][2dx+ux]
//   w3p [3][64][tap * 64 + c]                    value w3[o][c][dy][dx]
//   wfp [3][512][pixel * 64 + c]                 value wfc[o][c * P3 + pixel]
__device__ __forceinline__ void put3(bf16* dst, size_t plane, size_t i, float v)
{
    uint32_t a, b, c;
    x3_split2(v, 0.f, a, b, c);
    uint16_t* d = reinterpret_cast<uint16_t*>(dst);
    d[i] = (uint16_t)a; d[plane + i] = (uint16_t)b; d[2 * plane + i] = (uint16_t)c;
}
constexpr int kPackFloats = 8192;
struct LoadItem { const float* src; float* dst; int n; };
struct LoadParams {
    const float* wf;                    // [512][64 P3]
    float* wf_dst;
    LoadItem conv[2];                   // conv2, conv3: copied and packed
    LoadItem rest[9];                   // copied
    LoadItem turned[3];                 // conv1, conv2, conv3: [O][K] as [K][O]
    int turned_k[3];
    int P3;
    bf16 *w2p, *w3p, *wfp;              // nullptr: only copied
};
// One launch for all twelve tensors (a parameter update ends in one, so launches count: twelve copies and a packing pass
// took 45 us).  Blocks 0..511 take one row of the dense layer each and turn it through shared memory, sixteen bytes in and two
// channels of a pixel out at a time (four and two bytes before: 6.2 us for 84 x 84 x 4 and 10.3 for 128 x 128 x 4, calls in a row, now 4.1 and
// 5.6); the rest one element per thread.
__global__ void __launch_bounds__(256) load_fp32_kernel(const LoadParams p)
{
    __shared__ __align__(16) float s_row[kPackFloats];
    const int P3 = p.P3, F = 64 * P3;
    pdl_wait();
    if (blockIdx.x < 512) {
        const int o = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const bool vec = ((uintptr_t)p.wf & 15) == 0, fits = 4 * P3 <= kPackFloats;
        const int cstep = F <= kPackFloats || !fits ? 64 : kPackFloats / P3 / 4 * 4;    // channels per pass
        for (int c0 = 0; c0 < 64; c0 += cstep) {
            const int nc = c0 + cstep > 64 ? 64 - c0 : cstep, count = nc * P3;          // a multiple of four
            const size_t at = (size_t)o * F + (size_t)c0 * P3;
            if (vec)
                for (int i = threadIdx.x; i < count / 4; i += 256) {
                    const float4 v = reinterpret_cast<const float4*>(p.wf + at)[i];
                    reinterpret_cast<float4*>(p.wf_dst + at)[i] = v;
                    if (fits) reinterpret_cast<float4*>(s_row)[i] = v;
                }
            else
                for (int i = threadIdx.x; i < count; i += 256) {
                    const float v = p.wf[at + i];
                    p.wf_dst[at + i] = v;
                    if (fits) s_row[i] = v;
                }
            if (!p.wfp) continue;
            __syncthreads();
            const float* src = fits ? s_row : p.wf + at;
            uint32_t* dst = reinterpret_cast<uint32_t*>(p.wfp + (size_t)o * F + c0) + lane;
            const size_t plane = (size_t)256 * F;       // in pairs
            if (2 * lane < nc)
                for (int pix = warp; pix < P3; pix += 8) {                              // a lane: two channels
                    uint32_t a, b, c;
                    x3_split2(src[2 * lane * P3 + pix], src[(2 * lane + 1) * P3 + pix], a, b, c);
                    dst[pix * 32] = a; dst[plane + pix * 32] = b; dst[2 * plane + pix * 32] = c;
                }
            __syncthreads();
        }
        return;
    }
    int i = (blockIdx.x - 512) * 256 + threadIdx.x;
    if (i < 64 * 512) {
        const int o = i >> 9, k = i & 511, tap = k >> 7, cp = k & 127;
        const int dy = tap >> 1, dx = tap & 1, uy = cp >> 6, ux = (cp >> 5) & 1, c = cp & 31;
        if (p.w2p) put3(p.w2p, 64 * 512, i, p.conv[0].src[((o * 32 + c) * 4 + 2 * dy + uy) * 4 + 2 * dx + ux]);
        p.conv[0].dst[i] = p.conv[0].src[i];
        return;
    }
    i -= 64 * 512;
    if (i < 64 * 576) {
        const int o = i / 576, k = i - o * 576, tap = k >> 6, c = k & 63;
        if (p.w3p) put3(p.w3p, 64 * 576, i, p.conv[1].src[(o * 64 + c) * 9 + tap]);
        p.conv[1].dst[i] = p.conv[1].src[i];
        return;
    }
    i -= 64 * 576;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        if (i < p.rest[k].n) {
            p.rest[k].dst[i] = p.rest[k].src[i];
            return;
        }
        i -= p.rest[k].n;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (i < p.turned[k].n) {
            const int O = k == 0 ? 32 : 64;
            p.turned[k].dst[i] = p.turned[k].src[i % O * p.turned_k[k] + i / O];
            return;
        }
        i -= p.turned[k].n;
    }
}

// ---- heads ---------------------------------------------------------------------------------------------------
__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
    return v;
}

// One warp per sample: d J / d logits and d J / d value (dhead[i][0..A-1], dhead[i][A]), then the gradient of the
// hidden layer, dh[i][k] = (h[i][k] > 0) * sum_o dhead[i][o] whead[o][k], as three planes [n][512].
__global__ void __launch_bounds__(256)
head_backward_kernel(const float* __restrict__ logits, const float* __restrict__ values, const int32_t* __restrict__ actions,
                     const float* __restrict__ adv, const float* __restrict__ ret, const float* __restrict__ logp_old,
                     const float* __restrict__ whead, const float* __restrict__ h, float value_coef, float entropy_coef,
                     float clip, int n, int A, int* __restrict__ status, float* __restrict__ dhead, bf16* __restrict__ dh,
                     size_t dh_plane)
{
    extern __shared__ float4 s_w4[];                    // [A+1][512] head weights
    __shared__ float s_d[8][65];
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < (A + 1) * 128; i += 256) s_w4[i] = reinterpret_cast<const float4*>(whead)[i];
    pdl_wait();
    pdl_trigger();
    __syncthreads();
    const float inv_n = 1.0f / (float)n;
    for (int i = blockIdx.x + wib * gridDim.x; i < n; i += gridDim.x * 8) {      // few rows: a block each
        const int a = actions[i];
        const bool bad = (unsigned)a >= (unsigned)A;     // not used as an index: the row contributes nothing
        if (bad && lane == 0 && status) atomicCAS(status, 0, kStatusBadAction);
        float lg[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) lg[k] = lane + 32 * k < A ? logits[(size_t)i * A + lane + 32 * k] : -INFINITY;
        float m = fmaxf(lg[0], lg[1]);
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, k));
        float z = 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) z += lane + 32 * k < A ? expf(lg[k] - m) : 0.f;
        const float lse = m + logf(warp_sum(z));
        float lp[2], p[2], ent = 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bool in = lane + 32 * k < A;
            lp[k] = in ? lg[k] - lse : 0.f;
            p[k] = in ? expf(lp[k]) : 0.f;
            ent -= p[k] * lp[k];
        }
        ent = warp_sum(ent);
        float ds = adv[i];                               // d S_i / d log pi(a_i)
        if (logp_old && clip > 0.f && !bad) {
            const float lpa = __shfl_sync(0xffffffffu, a < 32 ? lp[0] : lp[1], a & 31);
            const float rho = expf(lpa - logp_old[i]);
            const float clipped = fminf(fmaxf(rho, 1.f - clip), 1.f + clip);
            ds = (rho * ds <= clipped * ds) ? rho * ds : 0.f;                  // the min takes its first argument
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int j = lane + 32 * k;
            // d log pi(a) / d logit_j = [j == a] - p_j ;   d H / d logit_j = -p_j (log p_j + H)
            if (j < A) s_d[wib][j] = bad ? 0.f : (ds * ((j == a ? 1.f : 0.f) - p[k]) - entropy_coef * p[k] * (lp[k] + ent)) * inv_n;
        }
        if (lane == 0) s_d[wib][A] = bad ? 0.f : 2.f * value_coef * (ret[i] - values[i]) * inv_n;
        __syncwarp();
        for (int j = lane; j <= A; j += 32) dhead[(size_t)i * (A + 1) + j] = s_d[wib][j];
        float acc[16];                                   // hidden units 128*q + 4*lane + {0..3}
#pragma unroll
        for (int k = 0; k < 16; ++k) acc[k] = 0.f;
        for (int o = 0; o <= A; ++o) {
            const float d = s_d[wib][o];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 w = s_w4[o * 128 + 32 * q + lane];
                acc[4 * q] = fmaf(d, w.x, acc[4 * q]); acc[4 * q + 1] = fmaf(d, w.y, acc[4 * q + 1]);
                acc[4 * q + 2] = fmaf(d, w.z, acc[4 * q + 2]); acc[4 * q + 3] = fmaf(d, w.w, acc[4 * q + 3]);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 hv = reinterpret_cast<const float4*>(h + (size_t)i * 512)[32 * q + lane];
            uint2 pl[3];
            x3_split2(hv.x > 0.f ? acc[4 * q] : 0.f, hv.y > 0.f ? acc[4 * q + 1] : 0.f, pl[0].x, pl[1].x, pl[2].x);
            x3_split2(hv.z > 0.f ? acc[4 * q + 2] : 0.f, hv.w > 0.f ? acc[4 * q + 3] : 0.f, pl[0].y, pl[1].y, pl[2].y);
#pragma unroll
            for (int k = 0; k < 3; ++k) reinterpret_cast<uint2*>(dh + k * dh_plane + (size_t)i * 512)[32 * q + lane] = pl[k];
        }
        __syncwarp();
    }
}

// Partial sums over a range of samples: row o <= A of the block's tile of outputs is sum_i dhead[i][o] h[i][k], row
// A + 1 is sum_i dh[i][k] (the dense bias); the head biases sum_i dhead[i][o] follow the 512 columns.
//   part [range][A + 2][513]
constexpr size_t kHeadRanges = 40;
constexpr int kHeadTile = 11;                            // outputs per block
constexpr int kHeadLeast = 16;                           // samples of a range, at least
__global__ void __launch_bounds__(256)
head_wgrad_kernel(const float* __restrict__ dhead, const float* __restrict__ h, const bf16* __restrict__ dh, size_t dh_plane,
                  int n, int A, int per_range, float* __restrict__ part)
{
    __shared__ float s_acc[4][64];
    const int k = blockIdx.x * 64 + (threadIdx.x & 63), sub = threadIdx.x >> 6;
    const int o0 = blockIdx.z * kHeadTile;
    const int i0 = blockIdx.y * per_range, i1 = min(n, i0 + per_range);
    pdl_wait();
    pdl_trigger();
    float acc[kHeadTile];
#pragma unroll
    for (int j = 0; j < kHeadTile; ++j) acc[j] = 0.f;
    for (int i = i0 + sub; i < i1; i += 4) {
        const float x = h[(size_t)i * 512 + k];
        const float* d = dhead + (size_t)i * (A + 1) + o0;
#pragma unroll
        for (int j = 0; j < kHeadTile; ++j) {
            if (o0 + j <= A) acc[j] = fmaf(d[j], x, acc[j]);
            else if (o0 + j == A + 1) {
                const bf16* g = dh + (size_t)i * 512 + k;
                acc[j] += x3_sum(__bfloat162float(g[0]), __bfloat162float(g[dh_plane]) + __bfloat162float(g[2 * dh_plane]));
            }
        }
    }
    float* out = part + ((size_t)blockIdx.y * (A + 2) + o0) * 513 + blockIdx.x * 64;
#pragma unroll
    for (int j = 0; j < kHeadTile; ++j) {
        if (o0 + j >= A + 2) break;
        s_acc[sub][threadIdx.x & 63] = acc[j];
        __syncthreads();
        if (threadIdx.x < 64) out[j * 513 + threadIdx.x] = (s_acc[0][threadIdx.x] + s_acc[1][threadIdx.x]) + (s_acc[2][threadIdx.x] + s_acc[3][threadIdx.x]);
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x < kHeadTile && o0 + threadIdx.x <= A) {
        float t = 0.f;
        for (int i = i0; i < i1; ++i) t += dhead[(size_t)i * (A + 1) + o0 + threadIdx.x];
        part[((size_t)blockIdx.y * (A + 2) + o0 + threadIdx.x) * 513 + 512] = t;
    }
}

// ---- sums over the ranges, in index order, into the caller's tensors -----------------------------------------------
struct ReduceParams {
    const float *c1, *c2, *c3, *b1, *b2, *b3, *head;     // partials
    int r1, r2, r3, r3_last, rh;                         // ranges (r3_last: of conv3's last tap)
    size_t g1, g2, g3;                                   // floats between group indices
    const float* fc;                                     // [512][pixel * 64 + c]
    int C, Cp, A, P3;
    const float *dhead, *h;                              // few samples: the heads' sums are taken here (n > 0), else from `head`
    const bf16* dh;
    size_t dh_plane;
    int n;
    hts_grads out;
};
// One kernel less while there are few samples.  Gradient of 84 x 84 x 4 frames, us, here / in a kernel of their own, with 2, 6, 18 and 32
// actions: 40 samples 97 / 101, 97 / 102, 99 / 105, 100 / 106; 80 samples 125 / 128, 126 / 129, 126 / 131, 127 / 131; 88 134 / 134, 134 / 136,
// 135 / 137, 136 / 137; 112 the same within 1 %; 128 160 / 153, 161 / 155, 162 / 156, 163 / 156.
constexpr int kHeadsInReduce = 80;
constexpr int kTurnFloats = 4096;
static_assert((kHeadsInReduce + 3 * kHeadLeast) / kHeadLeast * 256 <= kTurnFloats, "a sum's chains");
// Sixteen terms in flight.
template <class Term>
__device__ __forceinline__ float sum_terms(int lo, int hi, Term term)
{
    float acc = 0.f;
    for (int r = lo; r < hi; r += 16) {
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = r + i < hi ? term(r + i) : 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) acc += v[i];
    }
    return acc;
}
// Blocks 0..511 turn one row of the dense gradient each into the caller's column order (c * P3 + pixel): written by the
// contraction itself, 4-byte pieces P3 apart cost it 20 us.  The others sum, four threads of a block (64 apart) to a sum: a quarter
// of the ranges each, then the quarters in order: gradient without its forward pass of 512 frames of 72 x 96 x 16 260 -> 241 us, of 40 68 -> 64,
// of 80 of 84 x 84 x 4 72.3 -> 71.3 (one thread to a sum waited for up to 148 ranges, sixteen at a time).  The heads' sums come first:
// with their blocks last a gradient of 80 takes 131.5 us instead of 129.2.
__global__ void __launch_bounds__(256) reduce_kernel(const ReduceParams p)
{
    __shared__ float s_row[kTurnFloats];
    pdl_wait();
    pdl_trigger();
    if (blockIdx.x < 512) {
        const int F = 64 * p.P3;
        const float* src = p.fc + (size_t)blockIdx.x * F;
        float* dst = p.out.fc_w + (size_t)blockIdx.x * F;
        const int pstep = kTurnFloats / 65;              // pixels per pass, rows of 65 against bank conflicts
        for (int q0 = 0; q0 < p.P3; q0 += pstep) {
            const int nq = p.P3 - q0 < pstep ? p.P3 - q0 : pstep;
            for (int i = threadIdx.x; i < nq * 64; i += 256) s_row[(i >> 6) * 65 + (i & 63)] = src[(size_t)q0 * 64 + i];
            __syncthreads();
            for (int i = threadIdx.x; i < nq * 64; i += 256) {
                const int c = i / nq, q = i - c * nq;
                dst[(size_t)c * p.P3 + q0 + q] = s_row[q * 65 + c];
            }
            __syncthreads();
        }
        return;
    }
    int i = (blockIdx.x - 512) * 64 + (threadIdx.x & 63);
    const int n3 = 5 * 8192, n2 = 4 * 8192, n1 = p.Cp / 2 * 4096, nh = (p.A + 2) * 513;
    const float* src = nullptr;                          // what this thread's sum adds up, and where it goes
    float* dst = nullptr;
    int ranges = 0, ho = -1, hk = 0;
    size_t stride = 0;
    float scale = 1.f;
    if (i < nh) {                                        // first: with the longest chains of loads
        ho = i / 513; hk = i - ho * 513;
        src = p.head + i; ranges = p.rh; stride = (size_t)nh;
        if (ho == p.A + 1) dst = hk < 512 ? p.out.fc_b + hk : nullptr;
        else if (hk == 512) dst = ho < p.A ? p.out.pi_b + ho : p.out.v_b;
        else dst = ho < p.A ? p.out.pi_w + ho * 512 + hk : p.out.v_w + hk;
    } else if ((i -= nh) < n3) {                         // [tap pair][tap of the pair, c][o]
        const int gi = i >> 13, e = i & 8191, m = e >> 6, o = e & 63, b = m >> 6, c = m & 63;
        const int tap = gi < 4 ? 2 * gi + b : 7 + b;
        src = p.c3 + gi * p.g3 + e; ranges = gi == 4 ? p.r3_last : p.r3; stride = 8192;
        if (gi < 4 || b != 0) dst = p.out.conv3_w + (o * 64 + c) * 9 + tap;      // tap 7 belongs to pair 3
    } else if ((i -= n3) < n2) {                         // [tap][(uy, ux, c)][o]
        const int tap = i >> 13, e = i & 8191, cp = e >> 6, o = e & 63;
        const int dy = tap >> 1, dx = tap & 1, uy = cp >> 6, ux = (cp >> 5) & 1, c = cp & 31;
        src = p.c2 + tap * p.g2 + e; ranges = p.r2; stride = 8192;
        dst = p.out.conv2_w + ((o * 32 + c) * 4 + 2 * dy + uy) * 4 + 2 * dx + ux;
    } else if ((i -= n2) < n1) {                         // [64 columns of the cell, tap pair][tap, column][o]
        const int gi = i >> 12, e = i & 4095, m = e >> 5, o = e & 31;
        const int tap = (gi & 1) * 2 + (m >> 6), k = (gi >> 1) * 64 + (m & 63);
        const int c = k >> 4, uy = (k >> 2) & 3, ux = k & 3, dy = tap >> 1, dx = tap & 1;
        src = p.c1 + gi * p.g1 + e; ranges = p.r1; stride = 4096; scale = 1.0f / 255.0f;
        if (c < p.C) dst = p.out.conv1_w + ((o * p.C + c) * 8 + 4 * dy + uy) * 8 + 4 * dx + ux;
    } else if ((i -= n1) < 64) {
        src = p.b3 + i; ranges = p.r3; stride = 64; dst = p.out.conv3_b + i;
    } else if (i < 128) {
        src = p.b2 + i - 64; ranges = p.r2; stride = 64; dst = p.out.conv2_b + i - 64;
    } else if (i < 160) {
        src = p.b1 + i - 128; ranges = p.r1; stride = 32; dst = p.out.conv1_b + i - 128;
    }
    const int part = threadIdx.x >> 6, t = threadIdx.x & 63;
    const bool samples = ho >= 0 && p.n > 0;             // of this sum, not of its block
    if (dst && samples) {
        // As head_wgrad_kernel adds: chains of every fourth sample of kHeadLeast, products not rounded before they are added.
        constexpr int IN_FLIGHT = 2, EACH = kHeadLeast / 4;      // ranges; a chain's samples
#pragma unroll 1
        for (int q = 0; q * kHeadLeast < p.n; q += IN_FLIGHT) {
            float2 v[IN_FLIGHT * EACH];
#pragma unroll
            for (int k = 0; k < IN_FLIGHT * EACH; ++k) {
                const int r = q * kHeadLeast + 4 * k + part;
                v[k] = make_float2(0.f, 0.f);
                if (r >= p.n) continue;
                if (ho == p.A + 1) {
                    const bf16* g = p.dh + (size_t)r * 512 + hk;
                    v[k] = make_float2(1.f, x3_sum(__bfloat162float(g[0]), __bfloat162float(g[p.dh_plane]) + __bfloat162float(g[2 * p.dh_plane])));
                } else
                    v[k] = make_float2(p.dhead[(size_t)r * (p.A + 1) + ho], hk == 512 ? 1.f : p.h[(size_t)r * 512 + hk]);
            }
#pragma unroll
            for (int j = 0; j < IN_FLIGHT; ++j) {
                float acc = 0.f;
#pragma unroll
                for (int k = 0; k < EACH; ++k) acc = fmaf(v[j * EACH + k].x, v[j * EACH + k].y, acc);
                s_row[(q + j) * 256 + threadIdx.x] = acc;
            }
        }
    } else
        s_row[threadIdx.x] = dst ? sum_terms(ranges * part / 4, ranges * (part + 1) / 4, [&](int r) { return src[(size_t)r * stride]; }) : 0.f;
    __syncthreads();
    if (!dst || threadIdx.x >= 64) return;
    auto four = [&](int q) { const float* a = s_row + q * 256 + t; return (a[0] + a[64]) + (a[128] + a[192]); };
    float sum = four(0);
    if (samples) {                                       // the same quarters as of partial sums of kHeadLeast samples
        const int chains = (p.n + kHeadLeast - 1) / kHeadLeast;
        float q4[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            q4[q] = 0.f;
            for (int r = chains * q / 4; r < chains * (q + 1) / 4; ++r) q4[q] += four(r);
        }
        sum = (q4[0] + q4[1]) + (q4[2] + q4[3]);
    }
    *dst = sum * scale;
}

inline unsigned nblk(size_t total, int th) { return (unsigned)((total + th - 1) / th); }

}  // namespace

// Packed weights, workspace and tensor maps of the fp32-accurate network passes of one context.
struct X3State {
    Geometry g;
    int max_batch, Cp, H0, W0, G0, H1s, W1s, P1s, P2, P3;
    int sms;
    int* status;
    bool packed = false;                                 // the planes below hold the current weights
    bf16 *w2p = nullptr, *w3p = nullptr, *wfp = nullptr;
    // workspace
    bf16 *x0 = nullptr, *a1, *a2, *a3, *dh, *dz3, *dz2, *dz1;
    float *logits, *logp, *val, *ent, *dhead, *part1, *part2, *part3, *partf, *bias1, *bias2, *bias3, *headp;
    X3TapParams bfc, bc3, bc2;                           // batch-independent parts
    X3WgradParams wfc, wc3, wc2, wc1;
    CUtensorMap mW2, mW3, mWf;
    int mapped_n = 0;                                    // batch size the maps below were made for
    CUtensorMap mDh, mDz3, mDz2, vX0, vA1, vA2, vA3, vDh, vDz3, vDz2, vDz1;
};

namespace {

// A tap groups' slabs: one slab read at every tap's row offset, or, on very wide grids, a slab per tap.
bool wgrad_rings(X3WgradParams* p, int apl, int b_planes, int kr, int spread, int shared_slabs, int own_slabs, bool* shared)
{
    p->kr = kr;
    const int room = 227 * 1024 - 4 * 1024;
    for (int sh = 1; sh >= 0; --sh) {
        *shared = sh != 0;
        p->a_rows = sh ? kr + spread : kr;
        p->n_a = sh ? shared_slabs : own_slabs;
        if (p->a_rows > 256) continue;
        const int stage = p->n_a * ((apl * p->a_rows * 128 + 1023) & ~1023) + p->n_b * b_planes * kr * 128;
        p->stages = room / stage > 8 ? 8 : room / stage;
        if (p->stages >= (sh ? 2 : 1)) return true;
    }
    return false;
}

bool x3_plan(X3State* t)
{
    const Geometry& g = t->g;
    const int s1[4] = {0, 1, t->W0, t->W0 + 1}, s2[4] = {0, 1, t->W1s, t->W1s + 1}, n2[4] = {0, -1, -t->W1s, -t->W1s - 1};
    int s3[9], n3[9];
    const int zero = 0;
    for (int i = 0; i < 9; ++i) { s3[i] = (i / 3) * g.W2 + i % 3; n3[i] = -s3[i]; }
    auto tap = [&](X3TapParams& p, int mode, int chunks, int taps, const int* shift, int tap_cols, int n_tiles, int P, int W, int H_out,
                   int W_out, int P_dst, int W_dst, int pitch) {
        p = X3TapParams{};
        p.mode = mode; p.n_tiles = n_tiles; p.tap_cols = tap_cols; p.P = P; p.W = W; p.H_out = H_out; p.W_out = W_out;
        p.P_dst = P_dst; p.W_dst = W_dst; p.dst_pitch = pitch; p.status = t->status;
        return x3_taps_plan(&p, chunks, taps, shift);
    };
    if (!(tap(t->bfc, X3_DGRAD_FC, 8, 1, &zero, 0, t->P3, 1, 1, g.H3, g.W3, t->P2, g.W2, 64) &&
          tap(t->bc3, X3_DGRAD, 1, 9, n3, 64, 1, t->P2, g.W2, g.H2, g.W2, t->P1s, t->W1s, 64) &&
          tap(t->bc2, X3_DGRAD_S2D, 1, 4, n2, 128, 2, t->P1s, t->W1s, g.H1, g.W1, t->G0, t->W0, 128)))
        return false;

    bool sh;
    auto slab = [](const X3WgradParams& p, int apl) { return (apl * p.a_rows * 128 + 1023) & ~1023; };
    {   // dense layer: kind = (128 outputs, two pixels)
        X3WgradParams& p = t->wfc; p = X3WgradParams{};
        p.n_b = 2;
        if (!wgrad_rings(&p, 3, 3, kX3StageRows<64>, 0, 2, 2, &sh)) return false;
        p.ka = 4; p.a_step = 128; p.b_step = 128; p.slab_col[1] = 64;
        p.groups = 2; p.group_cap = 2; p.kinds = 4 * ((t->P3 + 1) / 2); p.ranges = p.last_ranges = 1;
        p.a_lbo[0] = p.a_lbo[1] = slab(p, 3); p.b_off[1] = 3 * p.kr * 128; p.P3 = t->P3;
    }
    {   // conv3: five pairs of taps (0,1) (2,3) (4,5) (6,7) (7,8)
        X3WgradParams& p = t->wc3; p = X3WgradParams{};
        p.n_b = 1;
        if (!wgrad_rings(&p, 3, 3, kX3StageRows<64>, s3[8], 1, 4, &sh)) return false;
        p.ka = 1; p.kinds = 3; p.group_mul = 2; p.groups = 2; p.group_cap = 5;
        for (int gi = 0; gi < 5; ++gi) {
            const int t0 = gi < 4 ? 2 * gi : 7;
            p.a_off[gi] = sh ? s3[t0] * 128 : (gi & 1) * 2 * slab(p, 3);
            p.a_lbo[gi] = sh ? (s3[t0 + 1] - s3[t0]) * 128 : slab(p, 3);
            if (!sh) for (int b = 0; b < 2; ++b) p.slab_row[2 * gi + b] = s3[t0 + b];
        }
        if (!sh) p.slab_mul = 4;
    }
    {   // conv2: a group = one tap, its two 64-channel slabs
        X3WgradParams& p = t->wc2; p = X3WgradParams{};
        p.n_b = 1;
        if (!wgrad_rings(&p, 3, 3, kX3StageRows<64>, s2[3], 2, 4, &sh)) return false;
        p.ka = 1; p.kinds = 2; p.group_mul = 2; p.groups = 2; p.group_cap = 4;
        for (int gi = 0; gi < 4; ++gi) {
            p.a_off[gi] = sh ? s2[gi] * 128 : (gi & 1) * 2 * slab(p, 3);
            p.a_lbo[gi] = slab(p, 3);
            if (!sh) for (int b = 0; b < 2; ++b) { p.slab_col[2 * gi + b] = 64 * b; p.slab_row[2 * gi + b] = s2[gi]; }
        }
        if (sh) p.slab_col[1] = 64; else p.slab_mul = 4;
    }
    {   // conv1: kind = 64 columns of a cell, groups = the tap pairs (0,1) (2,3)
        X3WgradParams& p = t->wc1; p = X3WgradParams{};
        p.n_b = 2;
        if (!wgrad_rings(&p, 1, 1, kX3StageRows<32>, s1[3], 1, 4, &sh)) return false;
        p.ka = p.kinds = t->Cp / 4; p.a_step = 64; p.group_mul = 2; p.groups = 2; p.group_cap = 2 * p.kinds;
        for (int gi = 0; gi < p.group_cap; ++gi) {
            p.a_off[gi] = sh ? s1[2 * (gi & 1)] * 128 : (gi & 1) * 2 * slab(p, 1);
            p.a_lbo[gi] = sh ? 128 : slab(p, 1);
        }
        if (!sh) for (int i = 0; i < 4; ++i) p.slab_row[i] = s1[i];
    }
    for (X3WgradParams* p : {&t->wfc, &t->wc3, &t->wc2, &t->wc1}) p->status = t->status;
    return true;
}

}  // namespace

hts_status x3_create(const Geometry& g, int max_batch, int* status, X3State** out)
{
    X3State* t = new (std::nothrow) X3State();
    if (!t) return HTS_ERR_ALLOC;
    t->g = g; t->max_batch = max_batch; t->status = status;
    t->Cp = (g.C + 3) / 4 * 4; t->H0 = g.H / 4; t->W0 = g.W / 4; t->G0 = t->H0 * t->W0;
    t->H1s = (g.H1 + 1) / 2; t->W1s = (g.W1 + 1) / 2; t->P1s = t->H1s * t->W1s; t->P2 = g.H2 * g.W2; t->P3 = g.H3 * g.W3;
    t->sms = device_sm_count(device_slot());
    if (!x3_plan(t)) { delete t; return HTS_ERR_SHAPE; }
    *out = t;
    return HTS_OK;
}

void x3_destroy(X3State* t) { delete t; }

hts_status x3_load_weights(X3State* t, const hts_weights& w, const RefWeights& d, cudaStream_t s)
{
    const int A = t->g.A;
    auto f = [](const void* p) { return static_cast<const float*>(p); };
    const LoadParams p{f(w.fc_w), d.wfc,
                       {{f(w.conv2_w), d.w2, 64 * 512}, {f(w.conv3_w), d.w3, 64 * 576}},
                       {{f(w.conv1_w), d.w1, 32 * 64 * t->g.C}, {f(w.conv1_b), d.b1, 32}, {f(w.conv2_b), d.b2, 64}, {f(w.conv3_b), d.b3, 64},
                        {f(w.fc_b), d.bfc, 512}, {f(w.pi_w), d.whead, A * 512}, {f(w.v_w), d.whead + A * 512, 512}, {f(w.pi_b), d.bhead, A},
                        {f(w.v_b), d.bhead + A, 1}},
                       {{f(w.conv1_w), d.w1k, 32 * 64 * t->g.C}, {f(w.conv2_w), d.w2k, 64 * 512}, {f(w.conv3_w), d.w3k, 64 * 576}},
                       {64 * t->g.C, 512, 576}, t->P3, t->w2p, t->w3p, t->wfp};
    t->packed = t->wfp != nullptr;
    int n = 64 * 512 + 64 * 576;
    for (const LoadItem& it : p.rest) n += it.n;
    for (const LoadItem& it : p.turned) n += it.n;
    HTS_CUDA(launch_pdl(load_fp32_kernel, dim3(512 + nblk(n, 256)), dim3(256), 0, s, p));
    note_launch();
    return HTS_OK;
}

namespace {

// One allocation for the packed weights and everything the passes keep between kernels, made by the first gradient.  Zeroed once: positions of a grid outside a layer's
// output extent and channels added to the frames are never written and have to read as zero.
hts_status x3_workspace(X3State* t, bool (*alloc)(void* ctx, void** p, size_t bytes), void* alloc_ctx, cudaStream_t s)
{
    if (t->x0) return HTS_OK;
    const Geometry& g = t->g;
    const size_t nb = (size_t)t->max_batch, A = g.A;
    const int r1 = t->sms / t->wc1.kinds < 1 ? 1 : t->sms / t->wc1.kinds;
    size_t total = 0;
    auto room = [&](size_t bytes) { const size_t at = total; total += (bytes + 1023) & ~(size_t)1023; return at; };
    const size_t o_x0 = room(2 * nb * t->G0 * 16 * t->Cp), o_a1 = room(6 * nb * t->P1s * 128), o_a2 = room(6 * nb * t->P2 * 64),
                 o_a3 = room(6 * nb * g.F), o_dh = room(6 * nb * 512), o_dz3 = room(6 * nb * t->P2 * 64), o_dz2 = room(6 * nb * t->P1s * 64),
                 o_dz1 = room(2 * nb * t->G0 * 128), zeroed = total;
    const size_t n2 = 64 * 512, n3 = 64 * 576, nf = (size_t)512 * g.F;
    const size_t o_w2 = room(6 * n2), o_w3 = room(6 * n3), o_wf = room(6 * nf), o_pf = room(4 * nf);
    const size_t o_lg = room(4 * nb * A), o_lp = room(4 * nb), o_v = room(4 * nb),
                 o_e = room(4 * nb), o_dhead = room(4 * nb * (A + 1)), o_p1 = room(4 * (size_t)2 * t->wc1.kinds * r1 * 4096),
                 o_p2 = room(4 * (size_t)4 * (t->sms / 2 + 1) * 8192), o_p3 = room(4 * (size_t)5 * (t->sms * 2 / 5 + 1) * 8192), o_b1 = room(4 * (size_t)t->sms * 32),
                 o_b2 = room(4 * (size_t)t->sms * 64), o_b3 = room(4 * (size_t)t->sms * 64), o_hd = room(4 * kHeadRanges * (A + 2) * 513);
    void* q = nullptr;
    if (!alloc(alloc_ctx, &q, total + 1024)) return HTS_ERR_ALLOC;
    uint8_t* b = reinterpret_cast<uint8_t*>(((uintptr_t)q + 1023) & ~(uintptr_t)1023);
    HTS_CUDA(cudaMemsetAsync(b, 0, zeroed, s));
    auto H = [&](size_t o) { return reinterpret_cast<bf16*>(b + o); };
    auto Fl = [&](size_t o) { return reinterpret_cast<float*>(b + o); };
    t->w2p = H(o_w2); t->w3p = H(o_w3); t->wfp = H(o_wf); t->partf = Fl(o_pf);
    if (!(x3_make_map(&t->mW2, t->w2p, 512, 64, 3, 512, n2, 64, 3) && x3_make_map(&t->mW3, t->w3p, 576, 64, 3, 576, n3, 64, 3) &&
          x3_make_map(&t->mWf, t->wfp, g.F, 512, 3, g.F, nf, 64, 3)))
        return HTS_ERR_CUDA;
    t->x0 = H(o_x0); t->a1 = H(o_a1); t->a2 = H(o_a2); t->a3 = H(o_a3); t->dh = H(o_dh); t->dz3 = H(o_dz3); t->dz2 = H(o_dz2); t->dz1 = H(o_dz1);
    t->logits = Fl(o_lg); t->logp = Fl(o_lp); t->val = Fl(o_v); t->ent = Fl(o_e); t->dhead = Fl(o_dhead);
    t->part1 = Fl(o_p1); t->part2 = Fl(o_p2); t->part3 = Fl(o_p3); t->bias1 = Fl(o_b1); t->bias2 = Fl(o_b2); t->bias3 = Fl(o_b3); t->headp = Fl(o_hd);
    return HTS_OK;
}

// Tensor maps end with the rows of this batch: what an earlier, larger batch left behind reads as zero.
bool x3_map_batch(X3State* t, int n)
{
    if (t->mapped_n == n) return true;
    const Geometry& g = t->g;
    const size_t nb = (size_t)t->max_batch, N = (size_t)n;
    auto map = [](CUtensorMap* m, const bf16* p, uint64_t cols, uint64_t rows, uint64_t planes, uint64_t plane, int box, int box_planes) {
        return x3_make_map(m, p, cols, rows, planes, cols, plane, (uint32_t)box, (uint32_t)box_planes);
    };
    const size_t p1 = nb * t->P1s * 128, p2 = nb * t->P2 * 64, p3 = nb * g.F, ph = nb * 512, pz2 = nb * t->P1s * 64, x = nb * t->G0 * 16 * t->Cp;
    const bool ok =
        map(&t->vX0, t->x0, 16 * t->Cp, N * t->G0, 1, x, t->wc1.a_rows, 1) &&
        map(&t->vA1, t->a1, 128, N * t->P1s, 3, p1, t->wc2.a_rows, 3) &&
        map(&t->vA2, t->a2, 64, N * t->P2, 3, p2, t->wc3.a_rows, 3) &&
        map(&t->vA3, t->a3, g.F, N, 3, p3, t->wfc.kr, 3) &&
        map(&t->mDh, t->dh, 512, N, 3, ph, t->bfc.entry_rows, 3) && map(&t->vDh, t->dh, 512, N, 3, ph, t->wfc.a_rows, 3) &&
        map(&t->mDz3, t->dz3, 64, N * t->P2, 3, p2, t->bc3.entry_rows, 3) && map(&t->vDz3, t->dz3, 64, N * t->P2, 3, p2, t->wc3.kr, 3) &&
        map(&t->mDz2, t->dz2, 64, N * t->P1s, 3, pz2, t->bc2.entry_rows, 3) && map(&t->vDz2, t->dz2, 64, N * t->P1s, 3, pz2, t->wc2.kr, 3) &&
        map(&t->vDz1, t->dz1, 128, N * t->G0, 1, nb * t->G0 * 128, t->wc1.kr, 1);
    t->mapped_n = ok ? n : 0;
    return ok;
}

hts_status launch_frames(const void* arg, cudaStream_t s)
{
    const FramesParams& p = *static_cast<const FramesParams*>(arg);
    HTS_CUDA(launch_pdl(frames_kernel, dim3(nblk(p.items, 256)), dim3(256), 0, s, p));
    note_launch();
    return HTS_OK;
}

inline int tiles_of(size_t rows) { return (int)((rows + 127) / 128); }

}  // namespace

hts_status x3_gradient(X3State* t, const RefWeights& w, const RefWorkspace& ws, Profiler& prof, const uint8_t* obs, const int32_t* actions, const float* adv, const float* ret,
                       const float* logp_old, float value_coef, float entropy_coef, float clip, int n, const hts_grads& out,
                       bool (*alloc)(void* ctx, void** p, size_t bytes), void* alloc_ctx, cudaStream_t s)
{
    const Geometry& g = t->g;
    hts_status st = x3_workspace(t, alloc, alloc_ctx, s);
    if (st != HTS_OK) return st;
    if (!x3_map_batch(t, n)) return HTS_ERR_CUDA;
    if (!t->packed) {                                    // weights loaded before the first gradient
        const hts_weights own{w.w1, w.b1, w.w2, w.b2, w.w3, w.b3, w.wfc, w.bfc, w.whead, w.bhead, w.whead + (size_t)g.A * 512, w.bhead + g.A};
        st = x3_load_weights(t, own, w, s);
        if (st != HTS_OK) return st;
    }
    const size_t nb = (size_t)t->max_batch, N = (size_t)n;
    const size_t p1 = nb * t->P1s * 128, p2 = nb * t->P2 * 64, p3 = nb * g.F, ph = nb * 512, pz2 = nb * t->P1s * 64;

    const FramesParams fp{obs, g.C, t->Cp, g.H, g.W, N * t->G0 * t->Cp, ((uintptr_t)obs & 3) == 0, t->x0,
                          N * g.H1 * ((g.W1 + 3) / 4) > (size_t)96 * t->sms};
    const RefPlanes planes{t->a1, t->a2, t->a3, p1, p2, p3, fp.beside ? launch_frames : nullptr, &fp};
    if (!fp.beside) st = launch_frames(&fp, s);
    if (st != HTS_OK) return st;
    st = ref_forward(g, w, ws, obs, Indexing{}, t->status, n, prof, s, &planes);
    if (st != HTS_OK) return st;
    st = launch_heads(ws.h, 1, 0, nullptr, w.whead, w.bhead, g.A, nullptr, nullptr, 0, 0, n, Indexing{}, t->status, nullptr, t->logp, t->val,
                      t->ent, t->logits, nullptr, s, actions, false);
    if (st != HTS_OK) return st;
    auto run = [&](X3TapParams p, size_t rows, bf16* dst, size_t dst_plane, const bf16* mask, int mask_pitch) {
        p.m_tiles = tiles_of(rows); p.n = n; p.dst = dst; p.dst_plane = dst_plane; p.mask = mask; p.mask_pitch = mask_pitch;
        return p;
    };

    // ---- heads and data gradients
    const int sms = t->sms;
    {
        const size_t smem = (size_t)(g.A + 1) * 2048;
        static OncePerDevice allowed;
        HTS_CUDA(allow_shared(head_backward_kernel, allowed, false));
        const int blocks = n < sms ? n : (int)nblk(N, 8) < sms ? sms : (int)nblk(N, 8) < 4 * sms ? (int)nblk(N, 8) : 4 * sms;
        HTS_CUDA(launch_pdl(head_backward_kernel, dim3(blocks), dim3(256), smem, s, t->logits, t->val, actions, adv, ret, logp_old, w.whead, ws.h,
                            value_coef, entropy_coef, clip, n, g.A, t->status, t->dhead, t->dh, ph));
        note_launch();
    }
    int per_range = (n + (int)kHeadRanges - 1) / (int)kHeadRanges;
    if (per_range < kHeadLeast) per_range = kHeadLeast;
    const int rh = (n + per_range - 1) / per_range;
    if (n > kHeadsInReduce) {
        HTS_CUDA(launch_pdl(head_wgrad_kernel, dim3(8, rh, nblk(g.A + 2, kHeadTile)), dim3(256), 0, s, t->dhead, ws.h, t->dh, ph, n, g.A, per_range,
                            t->headp));
        note_launch();
    }

    // ---- data and weight gradients: ranges of at least one stage of rows
    auto cut = [&](X3WgradParams p, size_t rows, int ranges, int last) {
        p.row_chunks = (int)((rows + p.kr - 1) / p.kr);
        ranges = ranges < 1 ? 1 : ranges; last = last < 1 ? 1 : last;
        p.ranges = ranges < p.row_chunks ? ranges : p.row_chunks;
        p.last_ranges = last < p.row_chunks ? last : p.row_chunks;
        return p;
    };
    // Passes that do not wait for each other share a launch.  Blocks, one to an SM: of the dense layer's data gradient two thirds of
    // the SMs' at most, then its weight gradient's 128 x 128 outputs follow as SMs become free; conv3's data gradient gets its share of
    // the work (58 %: 45 to 58 % are the same within 2 % where tiles do not quantise, 256 and 512 rows gain 4 and 2 % from it), in
    // equal rounds; conv1's and conv2's weight gradients share by rows x their cost per row.  Gradient without its forward pass, us,
    // one launch per pass / now: 84 x 84 x 4 at 5 rows 75 / 57, 80 98 / 73, 256 147 / 125, 512 221 / 184, 1024 341 / 318; 72 x 96 x 16 at
    // 40 93 / 71, 512 283 / 261.
    X3WgradParams q = cut(t->wfc, N, 1, 1);
    q.fc_w = t->partf;
    const X3TapParams df = run(t->bfc, N, t->dz3, p2, t->a3, g.F);
    const int tiles_f = df.m_tiles * df.n_tiles, share_f = sms * 2 / 3 < 1 ? 1 : sms * 2 / 3;
    st = x3_data_weights_launch(t->mDh, t->mWf, df, tiles_f < share_f ? tiles_f : share_f, t->vDh, t->vA3, q, s);
    if (st != HTS_OK) return st;
    const X3TapParams d3 = run(t->bc3, N * t->P2, t->dz2, pz2, t->a2, 64);
    const int share_3 = sms * 58 / 100 < 1 ? 1 : sms * 58 / 100, rounds = (d3.m_tiles + share_3 - 1) / share_3;
    const int blocks_3 = (d3.m_tiles + rounds - 1) / rounds, left = sms - blocks_3;
    X3WgradParams q3 = cut(t->wc3, N * t->P2, left * 2 / 5, left / 5);          // the last kind has one group of five
    q3.part = t->part3; q3.group_stride = (size_t)q3.ranges * 8192; q3.bias_part = t->bias3;
    st = x3_data_weights_launch(t->mDz3, t->mW3, d3, blocks_3, t->vA2, t->vDz3, q3, s);
    if (st != HTS_OK) return st;
    st = x3_dgrad_launch(t->mDz2, t->mW2, run(t->bc2, N * t->P1s, t->dz1, 32, t->a1, 128), s);
    if (st != HTS_OK) return st;
    const double cost2 = 5.4 * t->P1s, cost1 = (double)t->wc1.kinds * t->G0;    // 0.44 and 0.082 ns a row
    int n2 = (int)(sms * cost2 / (cost1 + cost2) + 0.5);
    X3WgradParams q2 = cut(t->wc2, N * t->P1s, n2 / 2, n2 / 2);
    q2.part = t->part2; q2.group_stride = (size_t)q2.ranges * 8192; q2.bias_part = t->bias2;
    n2 = 2 * q2.ranges;
    const int r1 = (sms - n2) / t->wc1.kinds;
    X3WgradParams q1 = cut(t->wc1, N * t->G0, r1, r1);
    q1.part = t->part1; q1.group_stride = (size_t)q1.ranges * 4096; q1.bias_part = t->bias1;
    st = x3_weights_launch(t->vA1, t->vDz2, q2, t->vX0, t->vDz1, q1, s);
    if (st != HTS_OK) return st;
    ReduceParams r{};
    r.c1 = t->part1; r.c2 = t->part2; r.c3 = t->part3; r.b1 = t->bias1; r.b2 = t->bias2; r.b3 = t->bias3; r.head = t->headp;
    r.r1 = q1.ranges; r.r2 = q2.ranges; r.r3 = q3.ranges; r.r3_last = q3.last_ranges; r.rh = rh;
    r.g1 = q1.group_stride; r.g2 = q2.group_stride; r.g3 = q3.group_stride;
    r.dhead = t->dhead; r.h = ws.h; r.dh = t->dh; r.dh_plane = ph; r.n = n > kHeadsInReduce ? 0 : n;
    r.fc = t->partf; r.P3 = t->P3; r.C = g.C; r.Cp = t->Cp; r.A = g.A; r.out = out;
    const size_t total = (size_t)9 * 8192 + (size_t)t->Cp / 2 * 4096 + (size_t)(g.A + 2) * 513 + 160;
    HTS_CUDA(launch_pdl(reduce_kernel, dim3(512 + nblk(total, 64)), dim3(256), 0, s, r));
    note_launch();
    return HTS_OK;
}

}  // namespace hts
