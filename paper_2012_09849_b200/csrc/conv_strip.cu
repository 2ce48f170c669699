// fp32 convolutions of the actor step in strips.
//
// A thread owns PX consecutive pixels of one output row (a strip) and OT channels; a block's warps own LG strips x 32 / LG groups of
// channels each.  The sums are those of the plain loop: one chain over (c, u, v) per output.  Of a filter row a strip needs
// (PX - 1) s + k inputs instead of k PX gathered ones, so shared memory holds raw rows, filled by bulk copies of one warp (an
// mbarrier per stage; all waits are bounded), and a thread reads 20 inputs and 16 weights for 144 multiply-adds (second layer)
// where 8 x 8 tiles read 32 and 32 for 128.  Bound: the fp32 pipes (80 % busy while the sums run: 57 to 62 TFLOP/s of
// the pipes' 72), then what a block spends on its first copies and its stores.  At 1024 observations of 84 x 84 x 4 the
// three layers take 131 / 100 / 78 us, in gathered tiles 150 / 151 / 101.  All channels of a stage are one straight run of instructions,
// so that the next channel's loads are under way during a channel's sums: with a loop over channels (first layer: filter rows) 133 /
// 107 / 80, and 60.3 instead of 57.1 us for a step of 80.
// Rows have an odd number of 16-byte pieces and, for stride 2, even and odd rows lie apart: eight output rows' inputs are in eight
// different sixteenths of the banks.  Copies issued by the computing warps cost 20 % (their address chains come before every
// stage's first sums), one copying warp with 16-byte asynchronous copies 10 to 20 us a layer (40 of them per stage and lane).
#include <climits>
#include "common.cuh"
#include "conv_strip.cuh"
#include "f32x2.cuh"
#include "tc_host.cuh"
#include "tc_ptx.cuh"
#include "x3_gemm.cuh"

namespace hts {
namespace {

struct StripPlan {
    int segs;                           // strips per output row
    int rows;                           // rows of a phase (bytes: of four input rows each) that a tile reads of a frame at most
    int pch, slot;                      // 16-byte pieces: of a row, of a frame's part of a stage
    int frames;                         // of a tile, at most
    int X;                              // pieces between the rows of two frames of a tile, besides
    int o_pitch;                        // floats between channels of the outputs in shared memory; 0: stored from registers
    int frame0;                         // frame of the map that is the batch's first
};
struct Strip { int q, rr, sx, e, i; };  // of a thread: strip and row of the batch, strip of the row, frame, row of the frame

// A named barrier among the computing warps.
__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
// One filter row of one channel: a strip's inputs x times the row's weights w[tap][OC].  A packed multiply-add takes 2 clocks
// of its scheduler if it shares an operand with the one before it and 3 if not (three pairs of registers, two banks), so the
// weights stay while the pixels pass, there and back: 64 to 70 TFLOP/s of multiply-adds
// alone, 58 to 62 with the input kept and the weights passing.
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

// A stage is CK channels of the inputs and their weights.  fp32: one box per frame of the tile, whose row r holds what the tile's
// output row r reads (of a second frame rows start before its first: those are filled with zeros).  Bytes: the rows of a frame and
// a channel that a tile reads follow one another in memory, four of them make a row here, a bulk copy each.  (A copy takes the
// copying unit 70 clocks, whatever its size: with one per channel, phase and frame the third layer took 11.5 / 83 us at 80 / 1024
// observations, with boxes 10.5 / 80.)
template <typename TIn, int KS, int S, int PX, int OT, int LG, int WS, int CK, int NST, int PER_SM>
__global__ void __launch_bounds__(32 * (WS * (S == 4 ? 32 : 64) / (32 / LG * OT) + 1), PER_SM)
conv_strip_kernel(const ConvParams p, const StripPlan t, const __grid_constant__ CUtensorMap map)
{
    constexpr bool U8 = sizeof(TIn) == 1;
    constexpr int OC = S == 4 ? 32 : 64, WO = OC / (32 / LG * OT), NC = WS * WO, SEGS = LG * WS, KK = KS * KS, HALO = (KS - 1) / S;
    constexpr int PH = U8 ? 1 : S, RW = (PX - 1) * S + KS;
    constexpr int WCH = CK * KK * OC / 4;                // 16-byte pieces of weights per stage
    extern __shared__ float4 s_dyn[];
    __shared__ uint64_t full[NST], freed[NST];
    __shared__ int abort_flag;
    float4* s4 = s_dyn + (-tc::smem_u32(s_dyn) & 127) / 16;                      // [NST][inputs of CK channels | weights]
    const int XCH = t.slot, GP = t.rows * t.pch, CP = PH * GP, STAGE = ((U8 ? CK * XCH : XCH) + WCH + 7) / 8 * 8;
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
        if (p.early) pdl_trigger();
        const int frames = rr1 / p.Ho - e0 + 1;
        auto rows_of = [&](int f, int* lo) {
            *lo = f == 0 ? rr0 - e0 * p.Ho : 0;
            return (f == frames - 1 ? rr1 - (e0 + f) * p.Ho : p.Ho - 1) - *lo + 1 + HALO;
        };
        uint32_t bytes = WCH * 16;                       // of a stage
        int lo;
        if constexpr (U8)
            for (int f = 0; f < frames; ++f) bytes += CK * rows_of(f, &lo) * t.pch * 16;
        else
            bytes += frames * CK * CP * 16;
        int st = 0;
#pragma unroll 1
        for (; st < stages; ++st) {
            const int slot = st % NST;
            if (st >= NST && !tc::mbar_wait_warp(freed + slot, (st / NST - 1) & 1, &abort_flag, p.status, 40)) break;
            float4* dst = s4 + slot * STAGE;
            if (lane == 0) {
                tc::mbar_arrive_expect_tx(full + slot, bytes);
                tc::bulk_load(dst + STAGE - WCH, p.wk + (size_t)st * CK * KK * OC, WCH * 16, full + slot);
            }
            __syncwarp();
            if constexpr (U8) {
                for (int u = lane; u < frames * CK; u += 32) {
                    const int cc = u % CK, f = u / CK, rows = rows_of(f, &lo);
                    const TIn* x = static_cast<const TIn*>(p.x) + (frame_of(p, e0 + f) * p.C + st * CK + cc) * p.xl.chan + (size_t)lo * 4 * p.W;
                    tc::bulk_load(dst + cc * XCH + ((e0 + f) * p.Ho + lo - rr0) * t.pch + f * t.X, x, rows * t.pch * 16, full + slot);
                }
            } else
                for (int f = lane; f < frames; f += 32)
                    tc::tma_load_5d(dst + f * t.X, &map, 0, rr0 - (e0 + f) * p.Ho, 0, st * CK, t.frame0 + e0 + f, full + slot);
        }
        if (st < stages) tc::let_copies_land();
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
    pdl_wait();                                          // here, so that the waits' limit does not count the kernel before
#pragma unroll 1
    for (int st = 0; st < stages; ++st) {
        const int slot = st % NST;
        if (!tc::mbar_wait_warp(full + slot, (st / NST) & 1, &abort_flag, p.status, 42)) {
            tc::let_copies_land();                       // the outputs pass through the ring
            break;                                       // strip_store's barriers are met all the same
        }
        const float4* in = s4 + slot * STAGE;
        const float* w = reinterpret_cast<const float*>(in + STAGE - WCH) + o_t;
#pragma unroll (U8 ? 1 : CK)
        for (int cc = 0; cc < CK; ++cc) {
            float x[(RW + 3) / 4 * 4];
            if constexpr (U8) {
                const uint32_t* x4 = reinterpret_cast<const uint32_t*>(in + cc * XCH) + x_at;
#pragma unroll 4
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
                    strip_load<RW>(x, x4 + u % S * GP + u / S * t.pch);
                    strip_row<KS, S, PX, OT, OC>(acc, x, w + u * KS * OC);
                }
                w += KK * OC;
            }
        }
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(freed + slot);
    }
    strip_store<PX, OT, NC>(p, t, acc, k, q0 + ws * LG + g <= last, o_t, q0, last, OC, reinterpret_cast<float*>(s4));
}

constexpr int kSharedPerSm = 227 * 1024;

// A form of strips: its tile, and where that lies in shared memory for one geometry.
template <typename TIn_, int KS_, int S_, int PX_, int OT_, int LG_, int WS_, int CK_, int NST_, int PER_SM_>
struct StripForm {
    typedef TIn_ TIn;
    static constexpr int KS = KS_, S = S_, PX = PX_, OT = OT_, LG = LG_, WS = WS_, CK = CK_, NST = NST_, PER_SM = PER_SM_;
    static constexpr bool U8 = sizeof(TIn) == 1;
    static constexpr int OC = S == 4 ? 32 : 64, NC = WS * OC / (32 / LG * OT), SEGS = LG * WS, HALO = (KS - 1) / S, PH = U8 ? 1 : S;
    // C channels of rows of `pch` pieces, outputs of Ho x Wo.  Shared memory without the stored outputs; 0: not a shape for it.
    static int plan(int C, int pch, int Ho, int Wo, StripPlan* t)
    {
        t->segs = (Wo + PX - 1) / PX;
        if (C % CK || (t->segs > 1 && PX * S % 4)) return 0;
        const int rt = t->segs == 1 ? SEGS : (SEGS - 1) / t->segs + 2;
        t->frames = (rt + Ho - 2) / Ho + 1;
        t->pch = pch; t->rows = rt + HALO; t->X = 0;
        long long stage;
        if (U8) {
            t->X = (HALO * pch + 7) / 8 * 8;
            // a last strip that ends past its row reads on into what follows
            const int reach = ((t->segs - 1) * PX * 4 + (PX - 1) * S + KS + (KS - 1) * pch * 4 + 15) / 16;
            t->slot = (rt - 1) * pch + (t->frames - 1) * t->X + (reach > (1 + HALO) * pch ? reach : (1 + HALO) * pch);
            stage = (long long)CK * t->slot;
        } else {
            if (pch > 64 || t->rows > 256) return 0;     // a box
            const int box = (CK * PH * t->rows * pch + 7) / 8 * 8;                // a copy lands on 128 bytes
            t->X = box;
            stage = t->slot = t->frames * box;
        }
        const long long smem = NST * 16 * ((stage + CK * KS * KS * OC / 4 + 7) / 8 * 8) + 128;
        return smem <= kSharedPerSm / PER_SM - 1024 - 128 ? (int)smem : 0;
    }
};

template <typename Form>
bool strip_map(const RowLayout& l, const float* x, int C, int H, int Ho, int Wo, size_t frames, CUtensorMap* map)
{
    StripPlan t{};
    return !Form::plan(C, l.pitch / 4, Ho, Wo, &t) ||
           tc::make_rows_map(map, x, l.pitch, l.phase / l.pitch, l.phases, C, frames, t.rows, Form::CK);
}

template <typename Form>
hts_status launch_strip(const ConvParams& p, const CUtensorMap* map, cudaStream_t s)
{
    StripPlan t{};
    int smem = Form::plan(p.C, Form::U8 ? p.W / 4 : p.xl.pitch / 4, p.Ho, p.Wo, &t);
    const long long total = (long long)p.n * p.Ho * t.segs;
    if (!smem || total > INT_MAX / 4) return HTS_ERR_UNSUPPORTED;
    t.frame0 = p.frame0;
    const bool direct = p.yl.pitch % 4 == 0 && p.yl.phase % 4 == 0 && p.yl.chan % 4 == 0 && (Form::PX % 4 == 0 || t.segs == 1);
    t.o_pitch = direct ? 0 : (t.rows - Form::HALO) * p.Wo;
    if (4 * t.o_pitch * Form::OC + 128 > smem) smem = 4 * t.o_pitch * Form::OC + 128;
    if (smem > kSharedPerSm / Form::PER_SM - 1024 - 128) return HTS_ERR_UNSUPPORTED;
    auto kernel = conv_strip_kernel<typename Form::TIn, Form::KS, Form::S, Form::PX, Form::OT, Form::LG, Form::WS, Form::CK, Form::NST, Form::PER_SM>;
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(kernel, allowed));
    HTS_CUDA(launch_pdl(kernel, dim3((unsigned)((total + Form::SEGS - 1) / Form::SEGS)), dim3(32 * (Form::NC + 1)), (size_t)smem, s, p, t,
                        map ? *map : CUtensorMap{}));
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

template <int PX, int OT, int LG, int WS, int CK, int NST, int PER_SM>
using Form1 = StripForm<uint8_t, 8, 4, PX, OT, LG, WS, CK, NST, PER_SM>;
template <int PX, int OT, int LG, int CK, int NST, int PER_SM>
using Form2 = StripForm<float, 4, 2, PX, OT, LG, 1, CK, NST, PER_SM>;
template <int PX, int OT, int LG, int CK, int NST, int PER_SM>
using Form3 = StripForm<float, 3, 1, PX, OT, LG, 1, CK, NST, PER_SM>;
typedef Form1<2, 4, 8, 2, 2, 2, 4> Few1;
typedef Form1<4, 8, 8, 4, 2, 2, 3> Many1;
typedef Form1<5, 8, 8, 4, 2, 2, 3> Five1;
typedef Form1<4, 8, 8, 4, 1, 2, 3> Odd1;                // an odd number of channels
typedef Form2<4, 2, 4, 8, 2, 2> Few2;
typedef Form2<4, 2, 4, 4, 2, 4> Thin2;                 // wide rows: Few2's stages do not fit
typedef Form2<9, 2, 4, 4, 2, 4> Some2n;                 // rows up to 9 pixels; else of strips of 10
typedef Form2<10, 2, 4, 4, 2, 4> Some2w;
typedef Form2<9, 4, 8, 4, 2, 3> Many2n;
typedef Form2<10, 4, 8, 2, 3, 3> Many2w;                // (four channels of three frames' boxes are too much for three blocks per SM)
typedef Form3<4, 2, 4, 16, 2, 2> Few3;
typedef Form3<4, 2, 4, 8, 3, 2> Thin3;
typedef Form3<7, 2, 4, 8, 2, 3> Some3n;                 // rows up to 7 pixels; else of strips of 8
typedef Form3<8, 2, 4, 8, 2, 3> Some3w;

bool make_strip_maps(const Geometry& g, const RefWorkspace& ws, size_t frames, StripMaps* m)
{
    auto two = [&](auto form, CUtensorMap* map) { return strip_map<decltype(form)>(ws.l1, ws.a1, 32, g.H1, g.H2, g.W2, frames, map); };
    auto three = [&](auto form, CUtensorMap* map) { return strip_map<decltype(form)>(ws.l2, ws.a2, 64, g.H2, g.H3, g.W3, frames, map); };
    return two(Few2{}, &m->few2) && two(Thin2{}, &m->thin2) && three(Few3{}, &m->few3) && three(Thin3{}, &m->thin3) &&
           (g.W2 <= 9 ? two(Some2n{}, &m->some2) && two(Many2n{}, &m->many2) : two(Some2w{}, &m->some2) && two(Many2w{}, &m->many2)) &&
           (g.W3 <= 7 ? three(Some3n{}, &m->some3) : three(Some3w{}, &m->some3));
}

// A form takes a time that steps with the blocks of the fullest SM.  84 x 84 x 4, us at 1, 2, 3, 4 ... blocks, and what that is
// about (first + each more):
//   first layer    2 pixels x 4 channels 5.9, 7.7, 10.0, .. 17.0 (6): 5.6 + 2.2      4 x 8  9.1, 15.0, .. 27 (4), 38.8 (6), 134 (22): 9.1 + 6
//     5 x 8: 11.5 + 8.2, where that saves a round (step of 50 frames of 72 x 96 x 16 73 -> 63 us, of 100 116 -> 106; 80: 85 / 98)
//   second   4 x 2  7.4, 10.9, 14.9: 7.4 + 3.7     a row x 2  11.3, 18.0, 25.5, 32.9: 11.3 + 7.0     a row x 4  16.7, 29.5, .. 56 (4), .. 107 (8): 16.7 + 12.5
//   third    4 x 2  8.6, 11.8, .. 21.2 (4): 8.6 + 4.2     a row x 2  10.2, 15.6, .. 27.2 (4), 44.7 (7), 80 (13): 10.1 + 5.8
// Rows that leave strips half empty are faster in 128 x 64 tiles once there are many: 49 + 26.5 us for each more per SM in the second
// layer, 51 + 28 in the third.  The lines above are of full strips; of the forms for wider rows and of many blocks 18.5 + 15.2 (row x 4), 12.5 + 7.8 and 11 + 7.1
// (row x 2), 7.4 + 4.6 and 8.6 + 5.2 (4 x 2).  Second / third layer, us, tiles / strips: 2048 frames of 52 x 52 x 4 (rows of 5 and 3
// pixels) 99 / 118, 52 / 60; 512 of 128 x 128 x 4 (14 and 12) 177 / 202, 132 / 148; of 144 x 144 x 4 (16 and 14) 200 / 224, 191 / 178.
// Few2 and Few3 have four stages of 8 and 16 channels (eight of 4 and 8 before: step of 16 32.9 us, now 32.3).
// (the tiles of policy_ref.cu: 12 to 16 at 16 frames, 26 / 31 / 22 at 80, 150 / 151 / 101 at 1024).  A small tile's block has a short
// chain of sums, a large one more of them for each load.
hts_status launch_conv_strip(const ConvParams& p, const StripMaps* maps, cudaStream_t s)
{
    if (!p.wk || ((uintptr_t)p.x & 15)) return HTS_ERR_UNSUPPORTED;
    hts_status st = HTS_ERR_UNSUPPORTED;
    if (p.s == 4) {
        const int few = 56 + 22 * (strip_blocks(p, Few1::PX, Few1::SEGS) - 1), many = 91 + 60 * (strip_blocks(p, Many1::PX, Many1::SEGS) - 1),
                  five = 115 + 82 * (strip_blocks(p, Five1::PX, Five1::SEGS) - 1);
        if (few < many && few < five) st = launch_strip<Few1>(p, nullptr, s);
        if (st == HTS_ERR_UNSUPPORTED && five < many) st = launch_strip<Five1>(p, nullptr, s);
        if (st == HTS_ERR_UNSUPPORTED) st = launch_strip<Many1>(p, nullptr, s);
        if (st == HTS_ERR_UNSUPPORTED) st = launch_strip<Odd1>(p, nullptr, s);
        return st;
    }
    if (!maps) return HTS_ERR_UNSUPPORTED;
    if (p.s == 2) {
        const bool narrow = p.Wo <= 9;
        const int px = narrow ? 9 : 10;
        const int few = 74 + 37 * (strip_blocks(p, 4, 4) - 1), some = 113 + 70 * (strip_blocks(p, px, 4) - 1), many = 167 + 125 * (strip_blocks(p, px, 8) - 1);
        const int strips = few >= many && some >= many ? (narrow ? many : 185 + 152 * (strip_blocks(p, px, 8) - 1))
                         : few >= some ? (narrow ? some : 125 + 78 * (strip_blocks(p, px, 4) - 1)) : 74 + 46 * (strip_blocks(p, 4, 4) - 1);
        if (conv_tiles_large(p) && 490 + 265 * (conv_large_tiles(p) - 1) < strips) return HTS_ERR_UNSUPPORTED;
        if (few >= many && some >= many) st = narrow ? launch_strip<Many2n>(p, &maps->many2, s) : launch_strip<Many2w>(p, &maps->many2, s);
        if (st == HTS_ERR_UNSUPPORTED && few >= some) st = narrow ? launch_strip<Some2n>(p, &maps->some2, s) : launch_strip<Some2w>(p, &maps->some2, s);
        if (st == HTS_ERR_UNSUPPORTED) st = launch_strip<Few2>(p, &maps->few2, s);
        return st == HTS_ERR_UNSUPPORTED ? launch_strip<Thin2>(p, &maps->thin2, s) : st;
    }
    const bool narrow = p.Wo <= 7;
    const int few = 86 + 42 * (strip_blocks(p, 4, 4) - 1), row_blocks = strip_blocks(p, narrow ? 7 : 8, 4), some = 101 + 58 * (row_blocks - 1);
    const int strips = few < some ? 86 + 52 * (strip_blocks(p, 4, 4) - 1) : narrow ? some : 110 + 71 * (row_blocks - 1);
    // Rows of one pixel leave three quarters of a strip idle: 12.6, 16.8, 21, 25.5 us at 1, 2, 3, 4 blocks per SM, in 64 x 32 tiles 16.3 (2), 18.9 (3 and 4).
    if (p.Wo == 1 && strip_blocks(p, 4, 4) >= 3) return HTS_ERR_UNSUPPORTED;
    if (conv_tiles_large(p) && 510 + 280 * (conv_large_tiles(p) - 1) < strips) return HTS_ERR_UNSUPPORTED;
    if (few >= some)
        st = narrow ? launch_strip<Some3n>(p, &maps->some3, s) : launch_strip<Some3w>(p, &maps->some3, s);
    if (st == HTS_ERR_UNSUPPORTED) st = launch_strip<Few3>(p, &maps->few3, s);
    return st == HTS_ERR_UNSUPPORTED ? launch_strip<Thin3>(p, &maps->thin3, s) : st;
}

}  // namespace hts
