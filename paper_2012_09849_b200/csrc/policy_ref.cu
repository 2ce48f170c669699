// fp32 CUDA-core path of the actor step: the check path (fp32 weights) of the policy-value
// network of Appendix F.1 / F.2.  Every output is one chain of fp32 multiply-adds in a fixed order, whatever the
// tile that computes it, so a row's bits do not depend on the batch around it.  A context's convolutions run in strips
// (conv_strip.cu); the tiles here take what those do not: weights in the caller's layout (the step that allocates nothing),
// frames that are not 16-byte aligned, rows too wide for shared memory or of a length that leaves strips half empty.
#include <new>
#include <type_traits>
#include "common.cuh"
#include "conv_strip.cuh"
#include "f32x2.cuh"
#include "fc_f32.cuh"
#include "x3_gemm.cuh"

namespace hts {

struct RefMaps { StripMaps strips; FcMaps fc; };

RefMaps* ref_maps_create(const Geometry& g, const RefWeights& w, const RefWorkspace& ws, size_t frames)
{
    RefMaps* m = new (std::nothrow) RefMaps();
    if (m && make_strip_maps(g, ws, frames, &m->strips) && make_fc_maps(ws.a3, w.wfc, g.F, frames, &m->fc)) return m;
    delete m;
    return nullptr;
}
void ref_maps_destroy(RefMaps* maps) { delete maps; }

namespace {

__device__ __forceinline__ float4 load4(const float* p, bool vec)
{
    return vec ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
}

// Where the next kernel may start.  Blocks of a dependent launch that become resident early all settle on the first SMs
// that have room and stay there, waiting, while the others get none: its work then runs unevenly.  So the convolutions
// and the dense layer of many rows let it start as they end (no trigger), which costs it no more than its prologue (with
// gathered tiles n = 40 / 160 / 256 / 1024: 96 / 194 / 241 / 587 us per step with triggers after the wait, 81 / 168 / 201 / 549 without).
// The dense layer of few rows, before the small heads, still triggers (0.5 us per step).
// y[e,o,i,j] = relu(b[o] + in_scale * sum_{c,u,v} w[o,c,u,v] x[e,c,i s+u,j s+v]), summed over (c, u, v) in ascending
// order.  Implicit GEMM: a block owns PX consecutive output pixels of the batch and OC channels and gathers PX x KC
// inputs and OC x KC weights per step into shared memory, one step ahead; a thread owns PXT pixels x OT channels.
// Bound: no unit alone.  Inputs are gathered four bytes at a time, weights turned through registers in every block and chunk, and
// shared memory reaches registers at 128 bytes per clock (a thread loads 4 (PXT + OT) bytes per PXT x OT multiply-adds): 28 to 44
// TFLOP/s where strips reach 47 to 54 (first / second / third layer of 1024 observations 150 / 151 / 101 us, 131 / 100 / 78 in strips).
// A thread's pixels are runs of four, so a step's inputs are two 16-byte loads.
template <typename TIn, int PXT, int OT, int WPX, int WO, int KC, int PER_SM>
__global__ void __launch_bounds__(32 * WPX * WO, PER_SM)
conv_tile_kernel(const ConvParams p)
{
    constexpr int NT = 32 * WPX * WO, PX = WPX * 8 * PXT, OC = WO * 4 * OT;
    constexpr bool U8 = std::is_same<TIn, uint8_t>::value;
    constexpr int NPX = PX > NT ? PX / NT : 1, KL = PX > NT ? 1 : NT / PX;       // pixels of a loading thread, threads along k
    constexpr int UNIT = U8 ? 4 : 1;                                              // inputs per load
    constexpr int NA = KC / UNIT / KL;                                            // loads per pixel of a loading thread
    constexpr int NW = OC * KC / 4 / NT;
    static_assert(NPX * NT == PX * KL && NA * UNIT * KL == KC && NW * 4 * NT == OC * KC, "block shape");
    extern __shared__ __align__(16) float s_mem[];
    float* sA = s_mem;                                  // [2][KC][PX]
    float* sW = s_mem + 2 * KC * PX;                    // [2][KC][OC]
    int* s_off = reinterpret_cast<int*>(sW + 2 * KC * OC);   // input offset of each load unit
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int K = p.C * p.k * p.k, P = p.Ho * p.Wo;
    const int total = p.n * P, o_base = blockIdx.y * OC;
    for (int u = tid; u < K / UNIT; u += NT) {
        const int kk = u * UNIT, c = kk / (p.k * p.k), r = kk - c * p.k * p.k, uu = r / p.k;
        s_off[u] = c * p.xl.chan + x_tap(p, uu) + (r - uu * p.k);
    }
    pdl_wait();
    const TIn* src[NPX];
#pragma unroll
    for (int q = 0; q < NPX; ++q) {
        // past the end of the batch: pixels from its start.  The last one for all would make a warp copy one word to 32
        // places, which takes 32 passes (conv3, n = 72: 40 us, 26 with distinct words).
        const int px = (blockIdx.x * PX + (NPX > 1 ? tid + NT * q : tid % PX)) % total;
        const int e = px / P, r = px - e * P, i = r / p.Wo, j = r - i * p.Wo;
        src[q] = static_cast<const TIn*>(p.x) + frame_of(p, e) * p.C * p.xl.chan + x_row(p, i) + j * p.s;
    }
    __syncthreads();
    const int kl = NPX > 1 ? 0 : tid / PX, pl = NPX > 1 ? tid : tid % PX;
    uint32_t ra[U8 ? NPX * NA : 1];
    float4 rw[NW];
    auto fetch = [&](int k0, int buf) {
        int off[NA];                                    // all of them first: a copy may not be moved across another one
#pragma unroll
        for (int a = 0; a < NA; ++a) off[a] = s_off[k0 / UNIT + kl * NA + a];
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            const int u = kl * NA + a;
#pragma unroll
            for (int q = 0; q < NPX; ++q) {
                const TIn* s = src[q] + off[a];
                if constexpr (U8) {
                    if (p.words) ra[q * NA + a] = *reinterpret_cast<const uint32_t*>(s);
                    else ra[q * NA + a] = s[0] | (uint32_t)s[1] << 8 | (uint32_t)s[2] << 16 | (uint32_t)s[3] << 24;
                } else
                    cp_async4((uint32_t)__cvta_generic_to_shared(sA + (buf * KC + u) * PX + pl + NT * q), s);
            }
        }
#pragma unroll
        for (int a = 0; a < NW; ++a) {
            const int u = a * NT + tid, o = u % OC, kq = u / OC;
            rw[a] = load4(p.w + (size_t)(o_base + o) * K + k0 + 4 * kq, p.w_vec);
        }
    };
    auto store = [&](int buf) {
        if constexpr (U8) {
#pragma unroll
            for (int q = 0; q < NPX; ++q)
#pragma unroll
                for (int a = 0; a < NA; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        sA[(buf * KC + (kl * NA + a) * 4 + b) * PX + pl + NT * q] = (float)((ra[q * NA + a] >> (8 * b)) & 0xffu);
        }
#pragma unroll
        for (int a = 0; a < NW; ++a) {
            const int u = a * NT + tid, o = u % OC, kq = u / OC;
            float* d = sW + (buf * KC + 4 * kq) * OC + o;
            d[0] = rw[a].x; d[OC] = rw[a].y; d[2 * OC] = rw[a].z; d[3 * OC] = rw[a].w;
        }
    };
    const int wp = warp % WPX, wo = warp / WPX, g = lane & 7, og = lane >> 3;
    static_assert(PXT % 4 == 0, "16-byte loads");
    const int px_t = wp * 8 * PXT + 4 * g, o_t = wo * 4 * OT + og * OT;          // pixels px_t + 32 (q / 4) + q % 4
    f32x2 acc[PXT][OT / 2];
#pragma unroll
    for (int q = 0; q < PXT; ++q)
#pragma unroll
        for (int j = 0; j < OT / 2; ++j) acc[q][j] = 0;
    const int chunks = K / KC;
    fetch(0, 0);
    store(0);
    cp_async_wait_all();
    __syncthreads();
    for (int c = 0; c < chunks; ++c) {
        const int buf = c & 1;
        if (c + 1 < chunks) fetch((c + 1) * KC, buf ^ 1);
#pragma unroll 16
        for (int kk = 0; kk < KC; ++kk) {
            const float* a = sA + (buf * KC + kk) * PX + px_t;
            const float* w = sW + (buf * KC + kk) * OC + o_t;
            f32x2 wv[OT / 2];
#pragma unroll
            for (int j = 0; j < OT / 2; j += 2) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(w + 2 * j);
                wv[j] = t.x; wv[j + 1] = t.y;
            }
            float4 xv[PXT / 4];
#pragma unroll
            for (int q = 0; q < PXT / 4; ++q) xv[q] = *reinterpret_cast<const float4*>(a + 32 * q);
#pragma unroll
            for (int q = 0; q < PXT; ++q) {
                const float4 x4 = xv[q / 4];
                const f32x2 xx = both(q % 4 == 0 ? x4.x : q % 4 == 1 ? x4.y : q % 4 == 2 ? x4.z : x4.w);
#pragma unroll
                for (int j = 0; j < OT / 2; ++j) fma2(acc[q][j], xx, wv[j]);
            }
        }
        if (c + 1 < chunks) {
            store(buf ^ 1);
            cp_async_wait_all();
            __syncthreads();
        }
    }
#pragma unroll
    for (int q = 0; q < PXT; ++q) {
        const int px = blockIdx.x * PX + px_t + 32 * (q / 4) + q % 4;
        if (px >= total) continue;
        const int e = px / P, r = px - e * P, i = p.y_rows ? r / p.Wo : 0, x = r - i * p.Wo;
        float v[OT];
#pragma unroll
        for (int j = 0; j < OT; ++j) {
            const float t = fmaf(lane_of(acc[q][j / 2], j & 1), p.in_scale, p.b[o_base + o_t + j]);
            v[j] = t > 0.f ? t : 0.f;
            p.y[((size_t)e * p.O + o_base + o_t + j) * p.yl.chan + y_row(p, i) + x] = v[j];
        }
        if (p.planes) {
            __nv_bfloat16* d = p.planes + plane_row(p, e, i, x) + o_base + o_t;
#pragma unroll
            for (int j = 0; j < OT; j += 4) {
                uint2 o0, o1, o2;
                x3_split2(v[j], v[j + 1], o0.x, o1.x, o2.x);
                x3_split2(v[j + 2], v[j + 3], o0.y, o1.y, o2.y);
                *reinterpret_cast<uint2*>(d + j) = o0;
                *reinterpret_cast<uint2*>(d + p.plane + j) = o1;
                *reinterpret_cast<uint2*>(d + 2 * p.plane + j) = o2;
            }
        }
    }
}

// The same sums for batches too small to fill the device with tiles: 16 pixels x 32 channels per block of 128 threads,
// 2 x 2 per thread, K in groups of 64, up to twelve of them in the ring.  The weights of the whole ring are requested
// first (up to 98 KB) and belong to the first group's copies: the first product waits for all of them, the others for
// their own inputs alone.  Inputs and weights stay in K order, four of it per load.  Bound: latency (n = 16, conv2 and
// conv3: one warp per scheduler, 0.93 instructions per clock, shared memory at half its rate, 14.5 us alone).
constexpr int kSmallK = 64, kSmallPitch = kSmallK + 4, kSmallPx = 16, kSmallOc = 32;
template <typename TIn>
__global__ void __launch_bounds__(128)
conv_small_kernel(const ConvParams p, int ring)
{
    constexpr bool U8 = std::is_same<TIn, uint8_t>::value;
    extern __shared__ __align__(16) float s_mem[];      // [ring][16 + 32][pitch]
    __shared__ const TIn* s_src[kSmallPx];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kk2 = p.k * p.k, K = p.C * kk2, P = p.Ho * p.Wo, groups = K / kSmallK;
    const int total = p.n * P, px0 = blockIdx.x * kSmallPx, o_base = blockIdx.y * kSmallOc;
    auto fetch_w = [&](int gr, int slot) {
        float* dst = s_mem + (slot * (kSmallPx + kSmallOc) + kSmallPx) * kSmallPitch;
#pragma unroll
        for (int a = 0; a < kSmallOc * kSmallK / 4 / 128; ++a) {
            const int u = a * 128 + tid, o = u >> 4, q = (u & 15) * 4;
            const float* src = p.w + (size_t)(o_base + o) * K + gr * kSmallK + q;
            const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + o * kSmallPitch + q);
            if (p.w_vec) cp_async16(d, src);
            else
                for (int i = 0; i < 4; ++i) cp_async4(d + 4 * i, src + i);
        }
    };
    auto fetch_x = [&](int gr, int slot) {
        float* dst = s_mem + slot * (kSmallPx + kSmallOc) * kSmallPitch;
        if constexpr (U8) {
#pragma unroll
            for (int a = 0; a < kSmallPx * kSmallK / 4 / 128; ++a) {
                const int u = a * 128 + tid, px = u >> 4, k = gr * kSmallK + (u & 15) * 4;
                const int c = k / kk2, r = k - c * kk2, uu = r / p.k;
                const TIn* s = s_src[px] + c * p.xl.chan + x_tap(p, uu) + (r - uu * p.k);
                uint32_t w;
                if (p.words) w = *reinterpret_cast<const uint32_t*>(s);
                else w = s[0] | (uint32_t)s[1] << 8 | (uint32_t)s[2] << 16 | (uint32_t)s[3] << 24;
                *reinterpret_cast<float4*>(dst + px * kSmallPitch + (u & 15) * 4) =
                    make_float4((float)(w & 0xffu), (float)((w >> 8) & 0xffu), (float)((w >> 16) & 0xffu), (float)(w >> 24));
            }
        } else {
            const int k = gr * kSmallK + (tid & 63), c = k / kk2, r = k - c * kk2, uu = r / p.k;
            const int off = c * p.xl.chan + x_tap(p, uu) + (r - uu * p.k);
#pragma unroll
            for (int a = 0; a < kSmallPx / 2; ++a) {
                const int px = 2 * a + (tid >> 6);
                cp_async4((uint32_t)__cvta_generic_to_shared(dst + px * kSmallPitch + (tid & 63)), s_src[px] + off);
            }
        }
    };
    pdl_wait();
    for (int g = 0; g < ring; ++g) fetch_w(g, g);
    if (tid < kSmallPx) {
        int px = px0 + tid;
        px = px < total ? px : total - 1;
        const int e = px / P, r = px - e * P, i = r / p.Wo, j = r - i * p.Wo;
        s_src[tid] = static_cast<const TIn*>(p.x) + frame_of(p, e) * p.C * p.xl.chan + x_row(p, i) + j * p.s;
    }
    __syncthreads();
    for (int g = 0; g < ring; ++g) {
        fetch_x(g, g);
        cp_async_commit();
    }
    const int g8 = lane & 7, og = lane >> 3, o_t = warp * 8 + og * 2;            // pixels g8, g8 + 8; channels o_t, o_t + 1
    float a00 = 0.f, a01 = 0.f, a10 = 0.f, a11 = 0.f;                            // [pixel][channel]
    for (int gr = 0, slot = 0; gr < groups; ++gr) {
        // groups still in flight may be as many as were requested after this one
        const int later = groups - 1 - gr < ring - 1 ? groups - 1 - gr : ring - 1;
        if (later >= 8) cp_async_wait<8>(); else if (later >= 4) cp_async_wait<4>(); else if (later >= 2) cp_async_wait<2>();
        else if (later == 1) cp_async_wait<1>(); else cp_async_wait<0>();
        __syncthreads();
        const float* x = s_mem + (slot * (kSmallPx + kSmallOc) + g8) * kSmallPitch;
        const float* w = s_mem + (slot * (kSmallPx + kSmallOc) + kSmallPx + o_t) * kSmallPitch;
#pragma unroll
        for (int k = 0; k < kSmallK; k += 4) {
            const float4 x0 = *reinterpret_cast<const float4*>(x + k), x1 = *reinterpret_cast<const float4*>(x + 8 * kSmallPitch + k);
            const float4 w0 = *reinterpret_cast<const float4*>(w + k), w1 = *reinterpret_cast<const float4*>(w + kSmallPitch + k);
            a00 = fmaf(w0.x, x0.x, a00); a01 = fmaf(w1.x, x0.x, a01); a10 = fmaf(w0.x, x1.x, a10); a11 = fmaf(w1.x, x1.x, a11);
            a00 = fmaf(w0.y, x0.y, a00); a01 = fmaf(w1.y, x0.y, a01); a10 = fmaf(w0.y, x1.y, a10); a11 = fmaf(w1.y, x1.y, a11);
            a00 = fmaf(w0.z, x0.z, a00); a01 = fmaf(w1.z, x0.z, a01); a10 = fmaf(w0.z, x1.z, a10); a11 = fmaf(w1.z, x1.z, a11);
            a00 = fmaf(w0.w, x0.w, a00); a01 = fmaf(w1.w, x0.w, a01); a10 = fmaf(w0.w, x1.w, a10); a11 = fmaf(w1.w, x1.w, a11);
        }
        if (gr + ring < groups) {
            __syncthreads();
            fetch_w(gr + ring, slot);
            fetch_x(gr + ring, slot);
        }
        cp_async_commit();
        slot = slot + 1 == ring ? 0 : slot + 1;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int px = px0 + g8 + 8 * q;
        if (px >= total) continue;
        const int e = px / P, r = px - e * P, i = p.y_rows ? r / p.Wo : 0, x = r - i * p.Wo, o = o_base + o_t;
        float v[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float t = fmaf(q ? (j ? a11 : a10) : (j ? a01 : a00), p.in_scale, p.b[o + j]);
            v[j] = t > 0.f ? t : 0.f;
            p.y[((size_t)e * p.O + o + j) * p.yl.chan + y_row(p, i) + x] = v[j];
        }
        if (p.planes) {
            uint32_t o0, o1, o2;
            x3_split2(v[0], v[1], o0, o1, o2);
            uint32_t* d = reinterpret_cast<uint32_t*>(p.planes + plane_row(p, e, i, x) + o);
            d[0] = o0; d[p.plane / 2] = o1; d[p.plane] = o2;
        }
    }
}

template <typename TIn>
hts_status launch_conv_small(const ConvParams& p, cudaStream_t s)
{
    const size_t px = (size_t)p.n * p.Ho * p.Wo, sms = (size_t)device_sm_count(device_slot());
    const size_t blocks = (px + kSmallPx - 1) / kSmallPx * (p.O / kSmallOc);
    // as many groups in flight as let all the blocks be resident at once (conv2, n = 32: 31 us where two blocks fit, 22)
    const int most = blocks <= sms ? 12 : blocks <= 2 * sms ? 8 : blocks <= 3 * sms ? 5 : blocks <= 4 * sms ? 4 : 3;
    const int groups = p.C * p.k * p.k / kSmallK, ring = groups < most ? groups : most;
    const int smem = ring * (kSmallPx + kSmallOc) * kSmallPitch * (int)sizeof(float);
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(conv_small_kernel<TIn>, allowed));
    HTS_CUDA(launch_pdl(conv_small_kernel<TIn>, dim3((unsigned)((px + kSmallPx - 1) / kSmallPx), (unsigned)(p.O / kSmallOc)), dim3(128),
                        (size_t)smem, s, p, ring));
    note_launch();
    return HTS_OK;
}

template <typename TIn, int PXT, int OT, int WPX, int WO, int KC, int PER_SM>
hts_status launch_conv_tile(const ConvParams& p, cudaStream_t s)
{
    constexpr int NT = 32 * WPX * WO, PX = WPX * 8 * PXT, OC = WO * 4 * OT;
    const int K = p.C * p.k * p.k;
    const size_t smem = sizeof(float) * (2 * KC * PX + 2 * KC * OC) + sizeof(int) * (size_t)(K / (std::is_same<TIn, uint8_t>::value ? 4 : 1));
    auto kernel = conv_tile_kernel<TIn, PXT, OT, WPX, WO, KC, PER_SM>;
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(kernel, allowed));
    const size_t px = (size_t)p.n * p.Ho * p.Wo;
    HTS_CUDA(launch_pdl(kernel, dim3((unsigned)((px + PX - 1) / PX), (unsigned)(p.O / OC)), dim3(NT), smem, s, p));
    note_launch();
    return HTS_OK;
}

// A form takes a time that steps with the blocks of the SM that has most (conv2, us at 1, 2, 3 ... per SM: latency form 15, 19, 23,
// 27; 64 x 32 tiles 25, 35, 48, 62, 74; 128 x 64 49, 75, 101).  The latency form pays up to three blocks per SM, two where it converts
// frames (17 against 15).  Large tiles: where rows leave strips half empty or do not fit (second / third layer of 200 frames of
// 48 x 1024 x 4 175 / 103 us, 259 / 144 in 64 x 32 tiles), and many unaligned frames.
template <typename TIn>
hts_status launch_conv(const ConvParams& p, const StripMaps* maps, cudaStream_t s)
{
    const hts_status strips = launch_conv_strip(p, maps, s);
    if (strips != HTS_ERR_UNSUPPORTED) return strips;
    constexpr bool U8 = std::is_same<TIn, uint8_t>::value;
    if (conv_tiles(p, kSmallPx, kSmallOc) <= (U8 ? 2 : 3)) return launch_conv_small<TIn>(p, s);
    if (!conv_tiles_large(p)) return launch_conv_tile<TIn, 4, 4, 2, 2, 32, 5>(p, s);
    if constexpr (U8) return launch_conv_tile<TIn, 8, 8, 4, 1, 16, 4>(p, s);
    else return launch_conv_tile<TIn, 8, 8, 2, 2, 16, 4>(p, s);
}

// h[e,o] = relu(b[o] + sum over lanes l of (chain of f = l, l+32, l+64, ...)), the 32 chains added as a binary tree
// over the lane number (halves first), for few rows (and callers without tensor maps, layers of 64 features; fc_f32.cu takes the others).  A warp owns
// TE rows x TO outputs and lane l runs chain l of all of them: both operands are contiguous across the lanes, so neither needs a
// transposition, and one transposing reduction closes the tree (at each level a lane keeps half of its values and gets its partner's
// share of them).  The block's rows of x and w go through a ring in shared memory, COLS columns at a time.  Bound: few rows by the latency
// of the weights: narrow tiles, deep ring; many by shared memory and the fp32 pipes: 8 x 8 per warp.
template <int TE, int TO, int WE, int WO, int STAGES, int COLS>
__global__ void __launch_bounds__(32 * WE * WO)
fc_chain_kernel(const float* __restrict__ x, const float* __restrict__ w, const float* __restrict__ b,
                float* __restrict__ h, int n, int F, bool w_vec)
{
    constexpr int NV = TE * TO, RX = TE * WE, RW = TO * WO, NT = 32 * WE * WO, Q = COLS / 4, UNITS = (RX + RW) * Q;   // 16-byte pieces of a row, of a stage
    extern __shared__ __align__(16) float s_mem[];      // [STAGES][RX + RW][COLS]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int we = warp % WE, wo = warp / WE;
    const int e0 = (blockIdx.y * WE + we) * TE, o0 = (blockIdx.x * WO + wo) * TO;
    pdl_wait();
    if constexpr (TE < 8) pdl_trigger();
    f32x2 acc[TE][TO / 2];
#pragma unroll
    for (int i = 0; i < TE; ++i)
#pragma unroll
        for (int j = 0; j < TO / 2; ++j) acc[i][j] = 0;
    auto fetch = [&](int f, int st) {
        float* dst = s_mem + st * (RX + RW) * COLS;
#pragma unroll
        for (int a = 0; a < (UNITS + NT - 1) / NT; ++a) {
            const int u = a * NT + threadIdx.x, r = u / Q, q = u % Q * 4;
            if (UNITS % NT && u >= UNITS) break;
            if (COLS > 64 && f + q >= F) continue;
            const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + r * COLS + q);
            if (r < RX) cp_async16(d, x + (size_t)min((int)(blockIdx.y * RX) + r, n - 1) * F + f + q);
            else {
                const float* src = w + (size_t)(blockIdx.x * RW + r - RX) * F + f + q;
                if (w_vec) cp_async16(d, src);
                else
                    for (int i = 0; i < 4; ++i) cp_async4(d + 4 * i, src + i);
            }
        }
    };
    const int steps = (F + COLS - 1) / COLS;             // F is a multiple of 64
#pragma unroll
    for (int s = 0; s < STAGES - 1; ++s) {
        if (s < steps) fetch(COLS * s, s);
        cp_async_commit();
    }
    for (int s = 0; s < steps; ++s) {
        cp_async_wait<STAGES - 2>();
        __syncthreads();                                // stage s has landed for every thread; stage s - 1 is free
        if (s + STAGES - 1 < steps) fetch(COLS * (s + STAGES - 1), (s + STAGES - 1) % STAGES);
        cp_async_commit();
        const float* xr = s_mem + (s % STAGES) * (RX + RW) * COLS + we * TE * COLS + lane;
        const float* wr = s_mem + (s % STAGES) * (RX + RW) * COLS + (RX + wo * TO) * COLS + lane;
#pragma unroll
        for (int c = 0; c < COLS; c += 64) {
            if (c > 0 && COLS * s + c >= F) break;
            float xv[2][TE], wv[2][TO];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
#pragma unroll
                for (int j = 0; j < TO; ++j) wv[k][j] = wr[COLS * j + c + 32 * k];
#pragma unroll
                for (int i = 0; i < TE; ++i) xv[k][i] = xr[COLS * i + c + 32 * k];
            }
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int i = 0; i < TE; ++i) {
                    const f32x2 xx = both(xv[k][i]);
#pragma unroll
                    for (int j = 0; j < TO / 2; ++j) fma2(acc[i][j], xx, pair(wv[k][2 * j], wv[k][2 * j + 1]));
                }
        }
    }
    float v[NV];
#pragma unroll
    for (int i = 0; i < TE; ++i)
#pragma unroll
        for (int j = 0; j < TO; ++j) v[i * TO + j] = lane_of(acc[i][j / 2], j & 1);
    int id = 0;                                         // (row, output) of v[0]
#pragma unroll
    for (int m = 16, len = NV / 2; m > 0; m >>= 1, len >>= 1) {
        if (len >= 1) {
            const bool up = lane & m;
#pragma unroll
            for (int k = 0; k < len; ++k) {
                const float send = up ? v[k] : v[k + len], keep = up ? v[k + len] : v[k];
                v[k] = keep + __shfl_xor_sync(0xffffffffu, send, m);
            }
            id += up ? len : 0;
        } else
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], m);
    }
    constexpr int LEFT = NV >= 32 ? NV / 32 : 1;
#pragma unroll
    for (int k = 0; k < LEFT; ++k) {
        const int e = e0 + (id + k) / TO, o = o0 + (id + k) % TO;
        const float r = v[k] + b[o];
        if (e < n && (NV >= 32 || (lane & (32 / NV - 1)) == 0)) h[(size_t)e * 512 + o] = r > 0.f ? r : 0.f;
    }
}

template <int TE, int TO, int WE, int WO, int STAGES, int COLS>
hts_status launch_fc_chain(const float* x, const float* w, const float* b, float* h, int n, int F, cudaStream_t s)
{
    constexpr int smem = STAGES * (TE * WE + TO * WO) * COLS * 4;
    auto kernel = fc_chain_kernel<TE, TO, WE, WO, STAGES, COLS>;
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(kernel, allowed));
    HTS_CUDA(launch_pdl(kernel, dim3(512 / (TO * WO), (unsigned)((n + TE * WE - 1) / (TE * WE))), dim3(32 * WE * WO), (size_t)smem, s,
                        x, w, b, h, n, F, ((uintptr_t)w & 15) == 0));
    note_launch();
    return HTS_OK;
}
// The form goes by the blocks (128 per 16 rows) of the SM that has most of them, k.  The fewer it has, the more each must have in
// flight and the less often its warps may meet: stages of 512 columns, three deep at k = 1 and two at k = 2 (both fill the shared
// memory), of 128 columns above (step at k = 1 / 2 / 3, 3136 features: 45.4 / 52.4 / 71.5 us with the first, 45.8 / 48.1 / 69.4 with the second,
// 47.7 / 50.7 / 64.3 with the third).  Where there are no boxes, one wide block per SM takes as long as five narrow ones (64 features, the
// layer of 2048 rows: 35 us narrow, 21 wide).  From k = 3 on boxes are faster (the layer alone, this / boxes: 16 rows 9.8 / 12.1 us, 32 rows
// 11.7 / 12.2, 40 rows 15.8 / 12.3).
hts_status launch_fc(const float* x, const float* w, const float* b, float* h, int n, int F, const RefWorkspace& ws, int* status, cudaStream_t s)
{
    const int sms = device_sm_count(device_slot());
    const long k = (128L * ((n + 15) / 16) + sms - 1) / sms;
    if (k == 1) return launch_fc_chain<4, 4, 4, 1, 3, 512>(x, w, b, h, n, F, s);
    if (k == 2) return launch_fc_chain<4, 4, 4, 1, 2, 512>(x, w, b, h, n, F, s);
    const hts_status st = ws.maps ? launch_fc_lanes({b, h, n, F, ws.row0, status}, ws.maps->fc, s) : HTS_ERR_UNSUPPORTED;
    if (st != HTS_ERR_UNSUPPORTED) return st;
    return k > 5 ? launch_fc_chain<8, 8, 4, 2, 4, 64>(x, w, b, h, n, F, s) : launch_fc_chain<4, 4, 4, 1, 4, 128>(x, w, b, h, n, F, s);
}

__global__ void __launch_bounds__(256) dense_rows_kernel(const float* __restrict__ x, const RowLayout l, int H, int W, size_t total, float* __restrict__ out)
{
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= total) return;
    const size_t row = i / W, c = row / H;
    const int y = (int)(row - c * H);
    out[i] = x[c * l.chan + y % l.phases * l.phase + y / l.phases * l.pitch + (int)(i - row * W)];
}

}  // namespace

hts_status launch_dense_rows(const float* x, const RowLayout& l, int channels, int H, int W, int n, float* out, cudaStream_t s)
{
    const size_t total = (size_t)n * channels * H * W;
    dense_rows_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(x, l, H, W, total, out);
    HTS_LAUNCH_CHECK("dense_rows");
    return HTS_OK;
}

// `planes`: also leave the three hidden convolution outputs as bf16 planes for the gradient.
hts_status ref_forward(const Geometry& g, const RefWeights& w, const RefWorkspace& ws,
                       const uint8_t* obs, const Indexing& ix, int* status, int n, Profiler& prof, cudaStream_t s,
                       const RefPlanes* planes)
{
    hts_status st;
    const StripMaps* maps = ws.maps ? &ws.maps->strips : nullptr;
    auto layer = [&](const void* x, const RowLayout& xl, const float* wt, const float* wk, const float* b, float* y, const RowLayout& yl, int C, int H,
                     int W, int O, int k, int stride, int Ho, int Wo) {
        ConvParams p{};
        p.x = x; p.xl = xl; p.w = wt; p.wk = wk; p.b = b; p.y = y; p.yl = yl; p.n = n; p.frame0 = ws.row0; p.C = C; p.H = H; p.W = W; p.O = O; p.k = k; p.s = stride; p.Ho = Ho; p.Wo = Wo;
        p.status = status; p.in_scale = 1.f; p.w_vec = ((uintptr_t)wt & 15) == 0; p.y_rows = yl.pitch != Wo || yl.phases != 1; p.words = ((uintptr_t)x & 3) == 0;
        return p;
    };
    prof.begin(K_CONV1, s);
    ConvParams c1 = layer(obs, rows_dense(g.H, g.W), w.w1, w.w1k, w.b1, ws.a1, ws.l1, g.C, g.H, g.W, 32, 8, 4, g.H1, g.W1);
    c1.in_scale = 1.0f / 255.0f; c1.slots = ix.slots; c1.pool = ix.pool;
    if (planes) { c1.planes = planes->a1; c1.plane = planes->p1; c1.s2d = c1.y_rows = true; c1.W_rows = (g.W1 + 1) / 2; c1.P_rows = (g.H1 + 1) / 2 * c1.W_rows; c1.early = planes->beside_conv1; }
    st = launch_conv<uint8_t>(c1, nullptr, s);
    if (st != HTS_OK) return st;
    prof.end(K_CONV1, s);
    if (planes && planes->beside_conv1) {
        st = planes->beside_conv1(planes->arg, s);
        if (st != HTS_OK) return st;
    }
    prof.begin(K_CONV2, s);
    ConvParams c2 = layer(ws.a1, ws.l1, w.w2, w.w2k, w.b2, ws.a2, ws.l2, 32, g.H1, g.W1, 64, 4, 2, g.H2, g.W2);
    if (planes) { c2.planes = planes->a2; c2.plane = planes->p2; c2.P_rows = g.H2 * g.W2; }
    st = launch_conv<float>(c2, maps, s);
    if (st != HTS_OK) return st;
    prof.end(K_CONV2, s);
    prof.begin(K_CONV3, s);
    ConvParams c3 = layer(ws.a2, ws.l2, w.w3, w.w3k, w.b3, ws.a3, rows_dense(g.H3, g.W3), 64, g.H2, g.W2, 64, 3, 1, g.H3, g.W3);
    if (planes) { c3.planes = planes->a3; c3.plane = planes->p3; c3.P_rows = g.H3 * g.W3; }
    st = launch_conv<float>(c3, maps, s);
    if (st != HTS_OK) return st;
    prof.end(K_CONV3, s);
    prof.begin(K_FC, s);
    st = launch_fc(ws.a3, w.wfc, w.bfc, ws.h, n, g.F, ws, status, s);
    if (st != HTS_OK) return st;
    prof.end(K_FC, s);
    return HTS_OK;
}

}  // namespace hts

// ---- actor step that allocates nothing ----------------------------------------------------------
// Scratch for hts_policy_step_noalloc: hidden activations of the four layers plus the stacked
// head weights, as floats.  It lives in the library image, so every GPU that loads the library
// carries these 4 MiB until the process exits.
namespace {
constexpr size_t kNoAllocFloats = size_t(1) << 20;
static __device__ __align__(256) float g_noalloc_scratch[kNoAllocFloats];
constexpr int kMaxDevices = 64;
float* g_noalloc_ptr[kMaxDevices] = {};       // device address of the array, looked up once per device
}  // namespace

extern "C" hts_status hts_policy_step_noalloc(const hts_net_desc* d, const hts_weights* w, const uint8_t* obs,
                                              const int32_t* env_ids, const int32_t* t_per_env, int32_t t,
                                              uint64_t seed, int32_t n, int32_t* actions, float* logp,
                                              float* values, float* entropy, float* logits_or_null,
                                              void* cuda_stream)
{
    using namespace hts;
    if (!d || !w || !obs || !env_ids || !actions || !logp || !values || !entropy) return HTS_ERR_INVALID_ARG;
    const void* const* wp = reinterpret_cast<const void* const*>(w);
    for (int i = 0; i < 12; ++i) if (!wp[i]) return HTS_ERR_INVALID_ARG;
    if (d->weight_dtype != HTS_DTYPE_FP32) return HTS_ERR_UNSUPPORTED;
    if (n < 1 || d->C < 1 || d->num_actions < 1 || d->num_actions > 64) return HTS_ERR_INVALID_ARG;
    if (d->H % 4 || d->W % 4 || d->H < 8 || d->W < 8) return HTS_ERR_SHAPE;
    Geometry g{};
    g.C = d->C; g.H = d->H; g.W = d->W; g.A = d->num_actions;
    g.H1 = conv_out(g.H, 8, 4); g.W1 = conv_out(g.W, 8, 4);
    if (g.H1 < 4 || g.W1 < 4) return HTS_ERR_SHAPE;
    g.H2 = conv_out(g.H1, 4, 2); g.W2 = conv_out(g.W1, 4, 2);
    if (g.H2 < 3 || g.W2 < 3) return HTS_ERR_SHAPE;
    g.H3 = conv_out(g.H2, 3, 1); g.W3 = conv_out(g.W2, 3, 1);
    g.F = 64 * g.H3 * g.W3;
    const size_t nn = (size_t)n;
    const size_t f_a1 = nn * 32 * g.H1 * g.W1, f_a2 = nn * 64 * g.H2 * g.W2, f_a3 = nn * g.F, f_h = nn * 512;
    const size_t f_wh = (size_t)(g.A + 1) * 512, f_bh = (size_t)g.A + 1;
    if (f_a1 + f_a2 + f_a3 + f_h + f_wh + f_bh > kNoAllocFloats) return HTS_ERR_INVALID_ARG;   // batch too large for the fixed scratch

    int dev = 0;
    HTS_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return HTS_ERR_UNSUPPORTED;
    if (!g_noalloc_ptr[dev]) {
        // In host code the array's name is only a handle: the kernels need its device address.
        float* ptr = nullptr;
        HTS_CUDA(cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_noalloc_scratch));
        g_noalloc_ptr[dev] = ptr;
    }
    float* base = g_noalloc_ptr[dev];
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const RefWorkspace ws{base, base + f_a1, base + f_a1 + f_a2, base + f_a1 + f_a2 + f_a3, rows_dense(g.H1, g.W1), rows_dense(g.H2, g.W2), nullptr, 0};
    float* whead = ws.h + f_h;
    float* bhead = whead + f_wh;
    // every scratch float is written before it is read, so nothing has to start at zero
    HTS_CUDA(cudaMemcpyAsync(whead, w->pi_w, (size_t)g.A * 512 * sizeof(float), cudaMemcpyDeviceToDevice, s));
    HTS_CUDA(cudaMemcpyAsync(whead + (size_t)g.A * 512, w->v_w, 512 * sizeof(float), cudaMemcpyDeviceToDevice, s));
    HTS_CUDA(cudaMemcpyAsync(bhead, w->pi_b, (size_t)g.A * sizeof(float), cudaMemcpyDeviceToDevice, s));
    HTS_CUDA(cudaMemcpyAsync(bhead + g.A, w->v_b, sizeof(float), cudaMemcpyDeviceToDevice, s));
    auto f = [](const void* p) { return const_cast<float*>(static_cast<const float*>(p)); };
    const RefWeights rw{f(w->conv1_w), f(w->conv1_b), f(w->conv2_w), f(w->conv2_b), f(w->conv3_w), f(w->conv3_b),
                        f(w->fc_w), f(w->fc_b), whead, bhead, nullptr, nullptr, nullptr};
    Profiler off;
    hts_status st = ref_forward(g, rw, ws, obs, Indexing{}, nullptr, n, off, s);
    if (st != HTS_OK) return st;
    return launch_heads(ws.h, 1, 0, nullptr, whead, bhead, g.A, env_ids, t_per_env, t, seed, n, Indexing{}, nullptr, actions,
                        logp, values, entropy, logits_or_null, nullptr, s, nullptr, false);
}
