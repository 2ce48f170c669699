// fp32 convolutions of the actor step in strips.
//
// A thread owns PX consecutive pixels of one output row (a strip) and OT channels; a block's warps own LG strips x 32 / LG groups of
// channels each.  The sums are those of the plain loop: one chain over (c, u, v) per output.  Of a filter row a strip needs
// (PX - 1) s + k inputs instead of k PX gathered ones, so shared memory holds raw rows, filled by bulk copies of one warp (an
// mbarrier per stage; all waits are bounded), and a thread reads 20 inputs and 16 weights for 144 multiply-adds (second layer)
// where 8 x 8 tiles read 32 and 32 for 128.  Bound: the fp32 pipes (80 % busy while the sums run; 60 TFLOP/s of the 70 that packed
// multiply-adds reach), then what a block spends on its first copies and its stores.  At 1024 observations of 84 x 84 x 4 the
// three layers take 134 / 104 / 83 us, in gathered tiles 150 / 151 / 101; at 80 15 / 17 / 11.5 against 26 / 31 / 22.
// Rows have an odd number of 16-byte pieces and, for stride 2, even and odd rows lie apart: eight output rows' inputs are in eight
// different sixteenths of the banks.  Copies issued by the computing warps cost 20 % (their address chains come before every
// stage's first sums), one copying warp with 16-byte asynchronous copies 10 to 20 us a layer (40 of them per stage and lane).
#include <climits>
#include "common.cuh"
#include "conv_strip.cuh"
#include "f32x2.cuh"
#include "tc_ptx.cuh"
#include "x3_gemm.cuh"

namespace hts {
namespace {

struct StripPlan {
    int segs;                           // strips per output row
    int pch, X, GP;                     // 16-byte pieces: row pitch, extra between frames, a phase of rows
    int o_pitch;                        // floats between channels of the outputs in shared memory; 0: stored from registers
};
struct Strip { int q, rr, sx, e, i; };  // of a thread: strip and row of the batch, strip of the row, frame, row of the frame

// A named barrier among the computing warps.
__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(tc::smem_u32(dst)), "l"(src), "r"(bytes), "r"(tc::smem_u32(bar)) : "memory");
}

// One filter row of one channel: a strip's inputs x times the row's weights w[tap][OC].  A packed multiply-add takes 2 clocks
// of its scheduler if it shares an operand with the one before it and 3 if not (three pairs of registers, two banks), so the
// weights stay while the pixels pass, there and back: 64 to 70 TFLOP/s, 58 to 62 with the input kept and the weights passing.
template <int KS, int S, int PX, int OT, int OC>
__device__ __forceinline__ void strip_row(f32x2 (&acc)[PX][OT / 2], const float (&x)[((PX - 1) * S + KS + 3) / 4 * 4], const float* w)
{
#pragma unroll
    for (int v = 0; v < KS; ++v) {
        f32x2 wv[OT / 2], xx[PX];
        if constexpr (OT >= 4) {
#pragma unroll
            for (int o = 0; o < OT / 2; o += 2) {
                const ulonglong2 two = *reinterpret_cast<const ulonglong2*>(w + v * OC + 2 * o);
                wv[o] = two.x; wv[o + 1] = two.y;
            }
        } else
            wv[0] = *reinterpret_cast<const f32x2*>(w + v * OC);
#pragma unroll
        for (int j = 0; j < PX; ++j) xx[j] = both(x[S * j + v]);
#pragma unroll
        for (int o = 0; o < OT / 2; ++o)
#pragma unroll
            for (int a = 0; a < PX; ++a) {
                const int j = o & 1 ? PX - 1 - a : a;
                fma2(acc[j][o], xx[j], wv[o]);
            }
    }
}

template <int RW>
__device__ __forceinline__ void strip_load(float (&x)[(RW + 3) / 4 * 4], const float4* x4)
{
#pragma unroll
    for (int a = 0; a < (RW + 3) / 4; ++a) {
        if (4 * a + 1 < RW) {
            const float4 v = x4[a];
            x[4 * a] = v.x; x[4 * a + 1] = v.y; x[4 * a + 2] = v.z; x[4 * a + 3] = v.w;
        } else
            x[4 * a] = reinterpret_cast<const float*>(x4 + a)[0];
    }
}
// Bytes become fp32 here: four lanes (of the four groups of channels) convert the same ones, but shared memory holds a quarter and
// frames are copied as they are.
template <int RW>
__device__ __forceinline__ void strip_load(float (&x)[(RW + 3) / 4 * 4], const uint32_t* x4)
{
#pragma unroll
    for (int a = 0; a < RW / 4; ++a) {
        const uint32_t v = x4[a];
#pragma unroll
        for (int b = 0; b < 4; ++b) x[4 * a + b] = (float)((v >> (8 * b)) & 0xffu);
    }
}

// A thread's sums into the caller's rows (and planes).  Rows of 16-byte pieces are stored from the registers, others through
// shared memory `s` of the NC computing warps, so that a warp writes whole sectors.
template <int PX, int OT, int NC>
__device__ __forceinline__ void strip_store(const ConvParams& p, const StripPlan& t, const f32x2 (&acc)[PX][OT / 2], const Strip& k, bool live,
                                            int o_t, int q0, int last, int n_oc, float* s)
{
    const int j0 = k.sx * PX, o0 = o_t, left = p.Wo - j0;
    float bias[OT];
#pragma unroll
    for (int o = 0; o < OT; ++o) bias[o] = p.b[o0 + o];
    auto value = [&](int j, int o) {
        const float v = fmaf(lane_of(acc[j][o / 2], o & 1), p.in_scale, bias[o]);
        return v > 0.f ? v : 0.f;
    };
    if (t.o_pitch == 0) {
        if (live) {
            float* y = p.y + ((size_t)k.e * p.O + o0) * p.yl.chan + y_row(p, k.i) + j0;
#pragma unroll
            for (int o = 0; o < OT; ++o) {
#pragma unroll
                for (int j = 0; j < PX; j += 4) {
                    if (j + 4 <= PX && j + 4 <= left)
                        *reinterpret_cast<float4*>(y + o * p.yl.chan + j) = make_float4(value(j, o), value(j + 1 < PX ? j + 1 : 0, o), value(j + 2 < PX ? j + 2 : 0, o), value(j + 3 < PX ? j + 3 : 0, o));
                    else
#pragma unroll
                        for (int a = j; a < j + 4 && a < PX; ++a)
                            if (a < left) y[o * p.yl.chan + a] = value(a, o);
                }
            }
        }
    } else {
        const int rr0 = q0 / t.segs, end = (last / t.segs - rr0) * p.Wo + min((last % t.segs + 1) * PX, p.Wo);
        bar_sync(15, 32 * NC);                           // nobody reads the ring any more
        if (live) {
            float* d = s + o_t * t.o_pitch + (k.rr - rr0) * p.Wo + j0;
#pragma unroll
            for (int o = 0; o < OT; ++o)
#pragma unroll
                for (int j = 0; j < PX; ++j)
                    if (j < left) d[o * t.o_pitch + j] = value(j, o);
        }
        bar_sync(15, 32 * NC);
        const int warp = threadIdx.x >> 5;
        for (int u = q0 % t.segs * PX + (threadIdx.x & 31); u < end; u += 32) {
            const int r = u / p.Wo, rr = rr0 + r, e = rr / p.Ho;
            float* y = p.y + (size_t)e * p.O * p.yl.chan + y_row(p, rr - e * p.Ho) + (u - r * p.Wo);
#pragma unroll 4
            for (int o = warp; o < n_oc; o += NC) y[(size_t)o * p.yl.chan] = s[o * t.o_pitch + u];
        }
    }
    if (p.planes && live) {
#pragma unroll
        for (int j = 0; j < PX; ++j) {
            if (j >= left) break;
            __nv_bfloat16* d = p.planes + plane_row(p, k.e, k.i, j0 + j) + o0;
            uint32_t o3[3][OT / 2];
#pragma unroll
            for (int o = 0; o < OT / 2; ++o) x3_split2(value(j, 2 * o), value(j, 2 * o + 1), o3[0][o], o3[1][o], o3[2][o]);
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                if constexpr (OT >= 8)
#pragma unroll
                    for (int o = 0; o < OT / 2; o += 4) *reinterpret_cast<uint4*>(d + l * p.plane + 2 * o) = make_uint4(o3[l][o], o3[l][o + 1], o3[l][o + 2], o3[l][o + 3]);
                else if constexpr (OT == 4) *reinterpret_cast<uint2*>(d + l * p.plane) = make_uint2(o3[l][0], o3[l][1]);
                else *reinterpret_cast<uint32_t*>(d + l * p.plane) = o3[l][0];
            }
        }
    }
}

// The rows of a frame, a channel and a phase that a tile reads follow one another in memory as they do in shared memory (bytes
// of frames: four rows make one), so a stage (CK channels) is a few bulk copies, one lane each, and one for its weights.
template <typename TIn, int KS, int S, int PX, int OT, int LG, int WS, int CK, int NST, int PER_SM>
__global__ void __launch_bounds__(32 * (WS * (S == 4 ? 32 : 64) / (32 / LG * OT) + 1), PER_SM)
conv_strip_kernel(const ConvParams p, const StripPlan t)
{
    constexpr bool U8 = sizeof(TIn) == 1;
    constexpr int OC = S == 4 ? 32 : 64, WO = OC / (32 / LG * OT), NC = WS * WO, SEGS = LG * WS, KK = KS * KS, HALO = (KS - 1) / S;
    constexpr int PH = U8 ? 1 : S, RW = (PX - 1) * S + KS;
    constexpr int WCH = CK * KK * OC / 4;                // 16-byte pieces of weights per stage
    extern __shared__ __align__(16) float4 s4[];         // [NST][inputs of CK channels | weights]
    __shared__ uint64_t full[NST], freed[NST];
    __shared__ int abort_flag;
    const int CP = PH * t.GP, XCH = CK * CP;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int total = p.n * p.Ho * t.segs, q0 = blockIdx.x * SEGS;
    const int rr0 = q0 / t.segs, last = min(q0 + SEGS, total) - 1, rr1 = last / t.segs;
    const int e0 = rr0 / p.Ho, stages = p.C / CK;
    if (tid == 0) {
        for (int i = 0; i < NST; ++i) { tc::mbar_init(full + i, 1); tc::mbar_init(freed + i, NC); }
        abort_flag = 0;
        tc::fence_barrier_init();
    }
    __syncthreads();
    if (warp == NC) {
        pdl_wait();
        const int frames = rr1 / p.Ho - e0 + 1, copies = frames * CK * PH;
        const size_t row = U8 ? 4 * p.W : p.xl.pitch;    // a row of t.pch pieces
        auto rows_of = [&](int f, int* lo) {
            *lo = f == 0 ? rr0 - e0 * p.Ho : 0;
            return (f == frames - 1 ? rr1 - (e0 + f) * p.Ho : p.Ho - 1) - *lo + 1 + HALO;
        };
        uint32_t bytes = WCH * 16;                       // of a stage
        int lo;
        for (int f = 0; f < frames; ++f) bytes += CK * PH * rows_of(f, &lo) * t.pch * 16;
        int st = 0;
#pragma unroll 1
        for (; st < stages; ++st) {
            const int slot = st % NST;
            if (st >= NST && !tc::mbar_wait_warp(freed + slot, (st / NST - 1) & 1, &abort_flag, p.status, 40)) break;
            float4* dst = s4 + slot * (XCH + WCH);
            if (lane == 0) {
                tc::mbar_arrive_expect_tx(full + slot, bytes);
                bulk_load(dst + XCH, p.wk + (size_t)st * CK * KK * OC, WCH * 16, full + slot);
            }
            __syncwarp();
            for (int u = lane; u < copies; u += 32) {
                const int ph = u % PH, cc = u / PH % CK, f = u / (PH * CK), rows = rows_of(f, &lo);
                const TIn* x = static_cast<const TIn*>(p.x) + (frame_of(p, e0 + f) * p.C + st * CK + cc) * p.xl.chan + ph * p.xl.phase + lo * row;
                bulk_load(dst + cc * CP + ph * t.GP + ((e0 + f) * p.Ho + lo - rr0) * t.pch + f * t.X, x, rows * t.pch * 16, full + slot);
            }
        }
        if (st < stages)                                 // given up: the copies in flight end before the block does
            for (int i = st < NST ? 0 : st - NST; i < st; ++i) tc::mbar_wait_warp(full + i % NST, (i / NST) & 1, &abort_flag, p.status, 41);
        return;
    }
    const int ws = warp % WS, wo = warp / WS, g = lane % LG, o_t = (wo * (32 / LG) + lane / LG) * OT;
    Strip k;
    k.q = min(q0 + ws * LG + g, last); k.rr = k.q / t.segs; k.sx = k.q - k.rr * t.segs; k.e = k.rr / p.Ho; k.i = k.rr - k.e * p.Ho;
    const int x_at = ((k.rr - rr0) * t.pch + (k.e - e0) * t.X) * (U8 ? 4 : 1) + k.sx * (PX * S / 4);
    f32x2 acc[PX][OT / 2];
#pragma unroll
    for (int j = 0; j < PX; ++j)
#pragma unroll
        for (int o = 0; o < OT / 2; ++o) acc[j][o] = 0;
#pragma unroll 1
    for (int st = 0; st < stages; ++st) {
        const int slot = st % NST;
        if (!tc::mbar_wait_warp(full + slot, (st / NST) & 1, &abort_flag, p.status, 42)) break;    // the barriers below are met all the same
        const float4* in = s4 + slot * (XCH + WCH);
        const float* w = reinterpret_cast<const float*>(in + XCH) + o_t;
#pragma unroll 1
        for (int cc = 0; cc < CK; ++cc) {
            float x[(RW + 3) / 4 * 4];
            if constexpr (U8) {
                const uint32_t* x4 = reinterpret_cast<const uint32_t*>(in + cc * CP) + x_at;
#pragma unroll 1
                for (int u = 0; u < KS; ++u) {
                    strip_load<RW>(x, x4);
                    strip_row<KS, S, PX, OT, OC>(acc, x, w);
                    x4 += p.W / 4;
                    w += KS * OC;
                }
            } else {
                const float4* x4 = in + cc * CP + x_at;
#pragma unroll
                for (int u = 0; u < KS; ++u) {
                    strip_load<RW>(x, x4 + u % S * t.GP + u / S * t.pch);
                    strip_row<KS, S, PX, OT, OC>(acc, x, w + u * KS * OC);
                }
                w += KK * OC;
            }
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(freed + slot);
    }
    pdl_wait();                                          // the kernel before may still read what this one writes
    strip_store<PX, OT, NC>(p, t, acc, k, q0 + ws * LG + g <= last, o_t, q0, last, OC, reinterpret_cast<float*>(s4));
}

constexpr size_t kSharedPerSm = 227 * 1024;
// The tile's place in shared memory.  HTS_ERR_UNSUPPORTED: not a shape for these strips.
template <typename TIn, int KS, int S, int PX, int OT, int LG, int WS, int CK, int NST, int PER_SM>
hts_status launch_strip(const ConvParams& p, cudaStream_t s)
{
    constexpr bool U8 = sizeof(TIn) == 1;
    constexpr int OC = S == 4 ? 32 : 64, NC = WS * OC / (32 / LG * OT), SEGS = LG * WS, HALO = (KS - 1) / S, RW = (PX - 1) * S + KS, PH = U8 ? 1 : S;
    StripPlan t{};
    t.segs = (p.Wo + PX - 1) / PX;
    if (p.C % CK || (t.segs > 1 && PX * S % 4)) return HTS_ERR_UNSUPPORTED;
    const long long total = (long long)p.n * p.Ho * t.segs;
    if (total > INT_MAX / 4) return HTS_ERR_UNSUPPORTED;
    t.pch = U8 ? p.W / 4 : p.xl.pitch / 4;
    t.X = (HALO * t.pch + 7) / 8 * 8;
    const int rt = t.segs == 1 ? SEGS : (SEGS - 1) / t.segs + 2, frames = (rt + p.Ho - 2) / p.Ho + 1;
    // a last strip that ends past its row reads on into what follows
    const int reach = U8 ? ((t.segs - 1) * PX * 4 + RW + (KS - 1) * p.W + 15) / 16 : ((t.segs - 1) * PX * S + RW + 3) / 4 + HALO * t.pch;
    t.GP = (rt - 1) * t.pch + (frames - 1) * t.X + (reach > (1 + HALO) * t.pch ? reach : (1 + HALO) * t.pch);
    const bool direct = p.yl.pitch % 4 == 0 && p.yl.phase % 4 == 0 && p.yl.chan % 4 == 0 && (PX % 4 == 0 || t.segs == 1);
    t.o_pitch = direct ? 0 : rt * p.Wo;
    size_t smem = 16 * NST * ((size_t)CK * KS * KS * OC / 4 + (size_t)CK * PH * t.GP);
    const size_t out = 4 * (size_t)t.o_pitch * OC;
    if (out > smem) smem = out;
    if (smem > kSharedPerSm / PER_SM - 1024 - 128) return HTS_ERR_UNSUPPORTED;
    auto kernel = conv_strip_kernel<TIn, KS, S, PX, OT, LG, WS, CK, NST, PER_SM>;
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(kernel, allowed));
    HTS_CUDA(launch_pdl(kernel, dim3((unsigned)((total + SEGS - 1) / SEGS)), dim3(32 * (NC + 1)), smem, s, p, t));
    note_launch();
    return HTS_OK;
}

}  // namespace

// Blocks of the fullest SM, if strips of px pixels go tile to a block.
static int strip_blocks(const ConvParams& p, int px, int tile)
{
    const long long strips = (long long)p.n * p.Ho * ((p.Wo + px - 1) / px), blocks = (strips + tile - 1) / tile;
    const int sms = device_sm_count(device_slot());
    return (int)((blocks + sms - 1) / sms);
}

// A form takes a time that steps with the blocks of the fullest SM.  84 x 84 x 4, us at 1, 2, 3, 4 ... blocks, and what that is
// about (first + each more):
//   first layer    2 pixels x 4 channels 5.9, 7.7, 10.0, .. 17.0 (6): 5.6 + 2.2      4 x 8  9.1, 15.0, .. 27 (4), 38.8 (6), 134 (22): 9.1 + 6
//   second   4 x 2  9.2, 11.1, 15.1: 9.2 + 3.7     a row x 2  11.6, 18.1, 25.0, 32.5: 11.6 + 6.8     a row x 4  17.1, 29.1, .. 55.4, .. 104 (8): 17.1 + 12.5
//   third    4 x 2  9.7, 12.6, .. 22.6 (4): 9.7 + 4.3     a row x 2  11.4, 16.7, .. 28.6 (4), 46.7 (7), 83 (13): 11.4 + 5.9
// (the tiles of policy_ref.cu: 12 to 16 at 16 frames, 26 / 31 / 22 at 80, 150 / 151 / 101 at 1024).  A small tile's block has a short
// chain of sums, a large one more of them for each load.
hts_status launch_conv_strip(const ConvParams& p, cudaStream_t s)
{
    if (!p.wk || ((uintptr_t)p.x & 15) || p.xl.pitch % 4) return HTS_ERR_UNSUPPORTED;
    hts_status st = HTS_ERR_UNSUPPORTED;
    if (p.s == 4) {
        if (p.C % 2 == 0 && 56 + 22 * (strip_blocks(p, 2, 16) - 1) < 91 + 60 * (strip_blocks(p, 4, 32) - 1))
            st = launch_strip<uint8_t, 8, 4, 2, 4, 8, 2, 2, 2, 4>(p, s);
        if (st == HTS_ERR_UNSUPPORTED) st = launch_strip<uint8_t, 8, 4, 4, 8, 8, 4, 2, 2, 3>(p, s);
        if (st == HTS_ERR_UNSUPPORTED) st = launch_strip<uint8_t, 8, 4, 4, 8, 8, 4, 1, 2, 3>(p, s);
        return st;
    }
    if (p.s == 2) {
        const int px = p.Wo <= 9 ? 9 : 10;
        const int few = 92 + 37 * (strip_blocks(p, 4, 4) - 1), some = 116 + 68 * (strip_blocks(p, px, 4) - 1), many = 171 + 125 * (strip_blocks(p, px, 8) - 1);
        if (few < some && few < many) st = launch_strip<float, 4, 2, 4, 2, 4, 1, 4, 3, 3>(p, s);
        else if (some < many) st = px == 9 ? launch_strip<float, 4, 2, 9, 2, 4, 1, 4, 2, 4>(p, s) : launch_strip<float, 4, 2, 10, 2, 4, 1, 4, 2, 4>(p, s);
        if (st == HTS_ERR_UNSUPPORTED) st = px == 9 ? launch_strip<float, 4, 2, 9, 4, 8, 1, 2, 3, 3>(p, s) : launch_strip<float, 4, 2, 10, 4, 8, 1, 2, 3, 3>(p, s);
        return st;
    }
    if (97 + 43 * (strip_blocks(p, 4, 4) - 1) < 114 + 59 * (strip_blocks(p, p.Wo <= 7 ? 7 : 8, 4) - 1)) st = launch_strip<float, 3, 1, 4, 2, 4, 1, 8, 3, 2>(p, s);
    if (st == HTS_ERR_UNSUPPORTED) st = p.Wo <= 7 ? launch_strip<float, 3, 1, 7, 2, 4, 1, 8, 2, 3>(p, s) : launch_strip<float, 3, 1, 8, 2, 4, 1, 8, 2, 3>(p, s);
    return st;
}

}  // namespace hts
