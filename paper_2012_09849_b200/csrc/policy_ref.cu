// fp32 CUDA-core path of the actor step: the check path (fp32 weights) of the policy-value
// network of Appendix F.1 / F.2.  Every output is one chain of fp32 multiply-adds in a fixed order, whatever the
// tile that computes it, so a row's bits do not depend on the batch around it.
#include <type_traits>
#include "common.cuh"
#include "x3_gemm.cuh"

namespace hts {
namespace {

__global__ void to_f32_kernel(const void* __restrict__ src, int dtype, float* __restrict__ dst, size_t count)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    dst[i] = (dtype == HTS_DTYPE_FP32) ? static_cast<const float*>(src)[i]
                                       : __bfloat162float(static_cast<const __nv_bfloat16*>(src)[i]);
}

typedef unsigned long long f32x2;                       // two fp32 lanes of a packed multiply-add
__device__ __forceinline__ void fma2(f32x2& acc, f32x2 a, f32x2 b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float lane_of(f32x2 v, int i) { return __uint_as_float(i ? (uint32_t)(v >> 32) : (uint32_t)v); }
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ float4 load4(const float* p, bool vec)
{
    return vec ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
}

struct ConvParams {
    const void* x;                      // [frames][C][H][W], u8 or fp32
    const float *w, *b;                 // [O][C k k], [O]
    float* y;                           // [n][O][Ho][Wo]
    int n, C, H, W, O, k, s, Ho, Wo;
    float in_scale;
    const int32_t* slots;               // frame of each row, or nullptr
    int pool;
    int* status;
    bool w_vec, words;                  // weights 16-byte aligned; frames 4-byte aligned
    __nv_bfloat16* planes;              // optional second output: three bf16 planes of pixel-major rows (x3_gemm.cuh)
    size_t plane;
    int W_rows, P_rows;                 // its grid; 2 x 2 pixels per row when s2d
    bool s2d;
};

// y[e,o,i,j] = relu(b[o] + in_scale * sum_{c,u,v} w[o,c,u,v] x[e,c,i s+u,j s+v]), summed over (c, u, v) in ascending
// order.  Implicit GEMM: a block owns PX consecutive output pixels of the batch and OC channels, gathers PX x KC inputs
// and OC x KC weights per step into shared memory (double-buffered; weights stored twice, as both lanes of a packed
// multiply-add), a thread owns PP pixel pairs x OT channels.  Bound: the fp32 pipes.  Packed multiply-adds reach
// 64 TFLOP/s in this pattern where scalar ones stop at 49 (three distinct registers per operation).
template <typename TIn, int PP, int OT, int WP, int WO, int KC, int PER_SM>
__global__ void __launch_bounds__(128, PER_SM)
conv_tile_kernel(const ConvParams p)
{
    constexpr int PX = WP * 16 * PP, OC = WO * 4 * OT;
    constexpr bool U8 = std::is_same<TIn, uint8_t>::value;
    constexpr int NPX = PX > 128 ? PX / 128 : 1, KL = PX > 128 ? 1 : 128 / PX;   // pixels of a loading thread, threads along k
    constexpr int UNIT = U8 ? 4 : 1;                                              // inputs per load
    constexpr int NA = KC / UNIT / KL;                                            // loads per pixel of a loading thread
    constexpr int NW = OC * KC / 4 / 128;
    static_assert(WP * WO == 4 && NA * UNIT * KL == KC && NW * 512 == OC * KC, "block shape");
    extern __shared__ __align__(16) float s_mem[];
    float* sA = s_mem;                                  // [2][KC][PX]
    float2* sW = reinterpret_cast<float2*>(s_mem + 2 * KC * PX);   // [2][KC][OC]
    int* s_off = reinterpret_cast<int*>(sW + 2 * KC * OC);         // input offset of each load unit
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int K = p.C * p.k * p.k, P = p.Ho * p.Wo;
    const int total = p.n * P, o_base = blockIdx.y * OC;
    for (int u = tid; u < K / UNIT; u += 128) {
        const int kk = u * UNIT, c = kk / (p.k * p.k), r = kk - c * p.k * p.k, uu = r / p.k;
        s_off[u] = (c * p.H + uu) * p.W + (r - uu * p.k);
    }
    pdl_wait();
    pdl_trigger();
    const TIn* src[NPX];
#pragma unroll
    for (int q = 0; q < NPX; ++q) {
        int px = blockIdx.x * PX + (NPX > 1 ? tid + 128 * q : tid % PX);
        px = px < total ? px : total - 1;
        const int e = px / P, r = px - e * P, i = r / p.Wo, j = r - i * p.Wo;
        size_t frame = (size_t)e;
        if (p.slots) {
            const int sl = p.slots[e];
            if ((unsigned)sl >= (unsigned)p.pool) { atomicCAS(p.status, 0, kStatusBadSlot); frame = 0; }
            else frame = (size_t)sl;
        }
        src[q] = static_cast<const TIn*>(p.x) + frame * p.C * p.H * p.W + (size_t)(i * p.s) * p.W + j * p.s;
    }
    __syncthreads();
    const int kl = NPX > 1 ? 0 : tid / PX, pl = tid % PX;
    uint32_t ra[U8 ? NPX * NA : 1];
    float4 rw[NW];
    auto fetch = [&](int k0, int buf) {
#pragma unroll
        for (int q = 0; q < NPX; ++q)
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                const int u = a * KL + kl;
                const TIn* s = src[q] + s_off[k0 / UNIT + u];
                if constexpr (U8) {
                    if (p.words) ra[q * NA + a] = *reinterpret_cast<const uint32_t*>(s);
                    else ra[q * NA + a] = s[0] | (uint32_t)s[1] << 8 | (uint32_t)s[2] << 16 | (uint32_t)s[3] << 24;
                } else
                    cp_async4((uint32_t)__cvta_generic_to_shared(sA + (buf * KC + u) * PX + pl + 128 * q), s);
            }
#pragma unroll
        for (int a = 0; a < NW; ++a) {
            const int u = a * 128 + tid, o = u % OC, kq = u / OC;
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
                        sA[(buf * KC + (a * KL + kl) * 4 + b) * PX + pl + 128 * q] = (float)((ra[q * NA + a] >> (8 * b)) & 0xffu);
        }
#pragma unroll
        for (int a = 0; a < NW; ++a) {
            const int u = a * 128 + tid, o = u % OC, kq = u / OC;
            float2* d = sW + (buf * KC + 4 * kq) * OC + o;
            d[0] = make_float2(rw[a].x, rw[a].x); d[OC] = make_float2(rw[a].y, rw[a].y);
            d[2 * OC] = make_float2(rw[a].z, rw[a].z); d[3 * OC] = make_float2(rw[a].w, rw[a].w);
        }
    };
    const int wp = warp % WP, wo = warp / WP, g = lane & 7, og = lane >> 3;
    const int px_t = wp * 16 * PP + 2 * g, o_t = wo * 4 * OT + og * OT;   // pairs at px_t + 16 q
    f32x2 acc[PP][OT];
#pragma unroll
    for (int q = 0; q < PP; ++q)
#pragma unroll
        for (int j = 0; j < OT; ++j) acc[q][j] = 0;
    fetch(0, 0);
    store(0);
    cp_async_wait();
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += KC, buf ^= 1) {
        const bool more = k0 + KC < K;
        if (more) fetch(k0 + KC, buf ^ 1);
#pragma unroll 8
        for (int kk = 0; kk < KC; ++kk) {
            f32x2 xv[PP], wv[OT];
            const float* a = sA + (buf * KC + kk) * PX + px_t;
            const float2* w = sW + (buf * KC + kk) * OC + o_t;
#pragma unroll
            for (int q = 0; q < PP; ++q) xv[q] = *reinterpret_cast<const f32x2*>(a + 16 * q);
#pragma unroll
            for (int j = 0; j < OT; j += 2) {
                const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(w + j);
                wv[j] = t.x; wv[j + 1] = t.y;
            }
#pragma unroll
            for (int q = 0; q < PP; ++q)
#pragma unroll
                for (int j = 0; j < OT; ++j) fma2(acc[q][j], xv[q], wv[j]);
        }
        if (more) {
            store(buf ^ 1);
            cp_async_wait();
            __syncthreads();
        }
    }
#pragma unroll
    for (int q = 0; q < PP; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int px = blockIdx.x * PX + px_t + 16 * q + h;
            if (px >= total) continue;
            const int e = px / P, r = px - e * P;
            float v[OT];
#pragma unroll
            for (int j = 0; j < OT; ++j) {
                const float t = fmaf(lane_of(acc[q][j], h), p.in_scale, p.b[o_base + o_t + j]);
                v[j] = t > 0.f ? t : 0.f;
                p.y[((size_t)e * p.O + o_base + o_t + j) * P + r] = v[j];
            }
            if (p.planes) {
                const int i = r / p.Wo, x = r - i * p.Wo;
                const size_t at = p.s2d ? ((size_t)e * p.P_rows + (size_t)(i >> 1) * p.W_rows + (x >> 1)) * 128 + ((i & 1) * 2 + (x & 1)) * 32
                                        : ((size_t)e * p.P_rows + r) * 64;
                uint32_t o0[OT / 2], o1[OT / 2], o2[OT / 2];
#pragma unroll
                for (int j = 0; j < OT / 2; ++j) x3_split2(v[2 * j], v[2 * j + 1], o0[j], o1[j], o2[j]);
                __nv_bfloat16* d = p.planes + at + o_base + o_t;
                if constexpr (OT == 8) {
                    *reinterpret_cast<uint4*>(d) = make_uint4(o0[0], o0[1], o0[2], o0[3]);
                    *reinterpret_cast<uint4*>(d + p.plane) = make_uint4(o1[0], o1[1], o1[2], o1[3]);
                    *reinterpret_cast<uint4*>(d + 2 * p.plane) = make_uint4(o2[0], o2[1], o2[2], o2[3]);
                } else {
#pragma unroll
                    for (int j = 0; j < OT / 2; ++j) {
                        reinterpret_cast<uint32_t*>(d)[j] = o0[j];
                        reinterpret_cast<uint32_t*>(d + p.plane)[j] = o1[j];
                        reinterpret_cast<uint32_t*>(d + 2 * p.plane)[j] = o2[j];
                    }
                }
            }
        }
}

template <typename TIn, int PP, int OT, int WP, int WO, int KC, int PER_SM>
hts_status launch_conv_tile(const ConvParams& p, cudaStream_t s)
{
    constexpr int PX = WP * 16 * PP, OC = WO * 4 * OT;
    const int K = p.C * p.k * p.k;
    const size_t smem = sizeof(float) * (2 * KC * PX + 4 * KC * OC) + sizeof(int) * (size_t)(K / (std::is_same<TIn, uint8_t>::value ? 4 : 1));
    auto kernel = conv_tile_kernel<TIn, PP, OT, WP, WO, KC, PER_SM>;
    static size_t smem_set_by_device[kDeviceSlots] = {};
    size_t& smem_set = smem_set_by_device[device_slot()];
    if (!smem_set || smem > smem_set) {
        HTS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        HTS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
        smem_set = smem;
    }
    const size_t px = (size_t)p.n * p.Ho * p.Wo;
    HTS_CUDA(launch_pdl(kernel, dim3((unsigned)((px + PX - 1) / PX), (unsigned)(p.O / OC)), dim3(128), smem, s, p));
    note_launch();
    return HTS_OK;
}

// The largest tile that still gives every SM two blocks: larger tiles load less per multiply-add, smaller ones
// spread a small batch over the device.
template <typename TIn>
hts_status launch_conv(const ConvParams& p, cudaStream_t s)
{
    const size_t px = (size_t)p.n * p.Ho * p.Wo, want = 2 * (size_t)device_sm_count(device_slot());
    if (p.O == 64 && px >= 128 * want) return launch_conv_tile<TIn, 4, 8, 2, 2, 16, 4>(p, s);
    if (p.O == 32 && px >= 256 * want) return launch_conv_tile<TIn, 4, 8, 4, 1, 16, 4>(p, s);
    if (px * p.O >= 64 * 32 * want) return launch_conv_tile<TIn, 2, 4, 2, 2, 32, 4>(p, s);
    return launch_conv_tile<TIn, 1, 2, 1, 4, 64, 4>(p, s);
}

// h[e,o] = relu(b[o] + sum over lanes l of (chain of f = l, l+32, l+64, ...)), the 32 chains added as a binary tree
// over the lane number (halves first).  512 threads: warp q runs chain q and then chain q + 16 for the block's whole
// TE x TO tile (a thread: PP row pairs x OT outputs), keeping the first result in shared memory; the tree closes
// across the warps.  Bound: the fp32 pipes for large batches, the weights' L2 traffic (block rows x 6.4 MB) below.
template <int PP, int OT, int PER_SM>
__global__ void __launch_bounds__(512, PER_SM)
fc_tile_kernel(const float* __restrict__ x, const float* __restrict__ w, const float* __restrict__ b,
               float* __restrict__ h, int n, int F, int O, bool w_vec)
{
    constexpr int TE = 16 * PP, TO = 4 * OT, NT = PP * OT * 2;
    constexpr int UX = TE * 8, UW = TO * 8;             // float4 loads per step of two chain elements (2 x 16 lanes)
    constexpr int NX = (UX + 511) / 512, NWL = (UW + 511) / 512;
    extern __shared__ __align__(16) float s_mem[];
    float* sX = s_mem;                                  // [2][32][TE], rows (element, lane), columns swizzled
    float2* sW = reinterpret_cast<float2*>(s_mem + 2 * 32 * TE);   // [2][32][TO]
    float* sH = reinterpret_cast<float*>(sW + 2 * 32 * TO);        // [NT][512], later [16][TE * TO]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane & 7, og = lane >> 3;
    const int e0 = blockIdx.y * TE, o0 = blockIdx.x * TO;
    constexpr int SX = TE >= 32 ? 3 : 1, SW = TO >= 32 ? 3 : 0;   // swizzle by groups of 8 columns
    float4 rx[NX], rw[NWL];
    // unit u: row r = u / 8, four lanes l4 = u % 4 of element (u / 4) % 2
    auto fetch = [&](int f0) {
#pragma unroll
        for (int a = 0; a < NX; ++a) {
            const int u = a * 512 + tid, r = u >> 3;
            if (UX % 512 == 0 || u < UX) rx[a] = *reinterpret_cast<const float4*>(x + (size_t)min(e0 + r, n - 1) * F + f0 + ((u >> 2) & 1) * 32 + (u & 3) * 4);
        }
#pragma unroll
        for (int a = 0; a < NWL; ++a) {
            const int u = a * 512 + tid, r = u >> 3;
            if (UW % 512 == 0 || u < UW) rw[a] = load4(w + (size_t)(o0 + r) * F + f0 + ((u >> 2) & 1) * 32 + (u & 3) * 4, w_vec);
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int a = 0; a < NX; ++a) {
            const int u = a * 512 + tid, r = u >> 3, row = ((u >> 2) & 1) * 16 + (u & 3) * 4;
            if (UX % 512 == 0 || u < UX) {
                float* d = sX + (buf * 32 + row) * TE + (r ^ ((u & SX) << 3));
                d[0] = rx[a].x; d[TE] = rx[a].y; d[2 * TE] = rx[a].z; d[3 * TE] = rx[a].w;
            }
        }
#pragma unroll
        for (int a = 0; a < NWL; ++a) {
            const int u = a * 512 + tid, r = u >> 3, row = ((u >> 2) & 1) * 16 + (u & 3) * 4;
            if (UW % 512 == 0 || u < UW) {
                float2* d = sW + (buf * 32 + row) * TO + (r ^ ((u & SW) << 3));
                d[0] = make_float2(rw[a].x, rw[a].x); d[TO] = make_float2(rw[a].y, rw[a].y);
                d[2 * TO] = make_float2(rw[a].z, rw[a].z); d[3 * TO] = make_float2(rw[a].w, rw[a].w);
            }
        }
    };
    pdl_wait();
    pdl_trigger();
    const int steps = F / 64;
    const int xs = ((warp >> 2) & SX) << 3, ws = ((warp >> 2) & SW) << 3;   // this warp's rows: lane group warp / 4
    f32x2 acc[PP][OT];
    for (int half = 0; half < 2; ++half) {
#pragma unroll
        for (int q = 0; q < PP; ++q)
#pragma unroll
            for (int j = 0; j < OT; ++j) acc[q][j] = 0;
        fetch(half * 16);
        __syncthreads();
        store(0);
        __syncthreads();
        for (int s = 0; s < steps; ++s) {
            if (s + 1 < steps) fetch((s + 1) * 64 + half * 16);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                f32x2 xv[PP], wv[OT];
                const float* xr = sX + ((s & 1) * 32 + i * 16 + warp) * TE;
                const float2* wr = sW + ((s & 1) * 32 + i * 16 + warp) * TO;
#pragma unroll
                for (int q = 0; q < PP; ++q) xv[q] = *reinterpret_cast<const f32x2*>(xr + ((16 * q + 2 * g) ^ xs));
#pragma unroll
                for (int j = 0; j < OT; j += 2) {
                    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(wr + ((og * OT + j) ^ ws));
                    wv[j] = t.x; wv[j + 1] = t.y;
                }
#pragma unroll
                for (int q = 0; q < PP; ++q)
#pragma unroll
                    for (int j = 0; j < OT; ++j) fma2(acc[q][j], xv[q], wv[j]);
            }
            if (s + 1 < steps) store((s + 1) & 1);
            __syncthreads();
        }
        if (half == 0) {
#pragma unroll
            for (int q = 0; q < PP; ++q)
#pragma unroll
                for (int j = 0; j < OT; ++j) {
                    sH[(2 * (q * OT + j)) * 512 + tid] = lane_of(acc[q][j], 0);
                    sH[(2 * (q * OT + j) + 1) * 512 + tid] = lane_of(acc[q][j], 1);
                }
        }
    }
    // level 16: chains q and q + 16, both of this thread; then one plane per warp for the levels 8, 4, 2, 1
    float v[NT];
#pragma unroll
    for (int q = 0; q < PP; ++q)
#pragma unroll
        for (int j = 0; j < OT; ++j) {
            const int i = 2 * (q * OT + j);
            v[i] = sH[i * 512 + tid] + lane_of(acc[q][j], 0);
            v[i + 1] = sH[(i + 1) * 512 + tid] + lane_of(acc[q][j], 1);
        }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < PP; ++q)
#pragma unroll
        for (int j = 0; j < OT; ++j)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh)
                sH[warp * (TE * TO) + (16 * q + 2 * g + hh) * TO + og * OT + j] = v[2 * (q * OT + j) + hh];
    __syncthreads();
    for (int i = tid; i < TE * TO; i += 512) {
        const int e = e0 + i / TO, o = o0 + i % TO;
        if (e >= n) break;
        float t[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) t[q] = sH[q * (TE * TO) + i];
#pragma unroll
        for (int m = 8; m > 0; m >>= 1)
#pragma unroll
            for (int q = 0; q < m; ++q) t[q] = t[q] + t[q + m];
        const float r = t[0] + b[o];
        h[(size_t)e * O + o] = r > 0.f ? r : 0.f;
    }
}

template <int PP, int OT, int PER_SM>
hts_status launch_fc_tile(const float* x, const float* w, const float* b, float* h, int n, int F, cudaStream_t s)
{
    constexpr int TE = 16 * PP, TO = 4 * OT;
    constexpr int smem = (2 * 32 * TE + 4 * 32 * TO + PP * OT * 2 * 512) * (int)sizeof(float);
    auto kernel = fc_tile_kernel<PP, OT, PER_SM>;
    static bool set_by_device[kDeviceSlots] = {};
    bool& set = set_by_device[device_slot()];
    if (!set) {
        HTS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        HTS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
        set = true;
    }
    HTS_CUDA(launch_pdl(kernel, dim3(512 / TO, (unsigned)((n + TE - 1) / TE)), dim3(512), (size_t)smem, s, x, w, b, h, n, F, 512,
                        ((uintptr_t)w & 15) == 0));
    note_launch();
    return HTS_OK;
}
hts_status launch_fc(const float* x, const float* w, const float* b, float* h, int n, int F, cudaStream_t s)
{
    if (n > 384) return launch_fc_tile<4, 8, 1>(x, w, b, h, n, F, s);
    if (n > 96) return launch_fc_tile<2, 4, 2>(x, w, b, h, n, F, s);
    return launch_fc_tile<1, 2, 2>(x, w, b, h, n, F, s);
}

inline unsigned blocks_for(size_t total, int threads) { return (unsigned)((total + threads - 1) / threads); }

}  // namespace

hts_status ref_convert_weights(const Geometry& g, int dtype, const hts_weights& src,
                               const RefWeights& dst, cudaStream_t s)
{
    struct Item { const void* p; float* q; size_t n; };
    const Item items[] = {
        {src.conv1_w, dst.w1, (size_t)32 * g.C * 64}, {src.conv1_b, dst.b1, 32},
        {src.conv2_w, dst.w2, (size_t)64 * 32 * 16},  {src.conv2_b, dst.b2, 64},
        {src.conv3_w, dst.w3, (size_t)64 * 64 * 9},   {src.conv3_b, dst.b3, 64},
        {src.fc_w, dst.wfc, (size_t)512 * g.F},       {src.fc_b, dst.bfc, 512},
        {src.pi_w, dst.whead, (size_t)g.A * 512},     {src.pi_b, dst.bhead, (size_t)g.A},
        {src.v_w, dst.whead + (size_t)g.A * 512, 512}, {src.v_b, dst.bhead + g.A, 1},
    };
    for (const Item& it : items) {
        to_f32_kernel<<<blocks_for(it.n, 256), 256, 0, s>>>(it.p, dtype, it.q, it.n);
        HTS_LAUNCH_CHECK("to_f32_kernel");
    }
    return HTS_OK;
}

// `planes`: also leave the three hidden convolution outputs as bf16 planes for the gradient.
hts_status ref_forward(const Geometry& g, const RefWeights& w, const RefWorkspace& ws,
                       const uint8_t* obs, const Indexing& ix, int* status, int n, Profiler& prof, cudaStream_t s,
                       const RefPlanes* planes)
{
    hts_status st;
    auto layer = [&](const void* x, const float* wt, const float* b, float* y, int C, int H, int W, int O, int k, int stride, int Ho, int Wo) {
        ConvParams p{};
        p.x = x; p.w = wt; p.b = b; p.y = y; p.n = n; p.C = C; p.H = H; p.W = W; p.O = O; p.k = k; p.s = stride; p.Ho = Ho; p.Wo = Wo;
        p.in_scale = 1.f; p.w_vec = ((uintptr_t)wt & 15) == 0; p.words = ((uintptr_t)x & 3) == 0;
        return p;
    };
    prof.begin(K_CONV1, s);
    ConvParams c1 = layer(obs, w.w1, w.b1, ws.a1, g.C, g.H, g.W, 32, 8, 4, g.H1, g.W1);
    c1.in_scale = 1.0f / 255.0f; c1.slots = ix.slots; c1.pool = ix.pool; c1.status = status;
    if (planes) { c1.planes = planes->a1; c1.plane = planes->p1; c1.s2d = true; c1.W_rows = (g.W1 + 1) / 2; c1.P_rows = (g.H1 + 1) / 2 * c1.W_rows; }
    st = launch_conv<uint8_t>(c1, s);
    if (st != HTS_OK) return st;
    prof.end(K_CONV1, s);
    prof.begin(K_CONV2, s);
    ConvParams c2 = layer(ws.a1, w.w2, w.b2, ws.a2, 32, g.H1, g.W1, 64, 4, 2, g.H2, g.W2);
    if (planes) { c2.planes = planes->a2; c2.plane = planes->p2; c2.P_rows = g.H2 * g.W2; }
    st = launch_conv<float>(c2, s);
    if (st != HTS_OK) return st;
    prof.end(K_CONV2, s);
    prof.begin(K_CONV3, s);
    ConvParams c3 = layer(ws.a2, w.w3, w.b3, ws.a3, 64, g.H2, g.W2, 64, 3, 1, g.H3, g.W3);
    if (planes) { c3.planes = planes->a3; c3.plane = planes->p3; c3.P_rows = g.H3 * g.W3; }
    st = launch_conv<float>(c3, s);
    if (st != HTS_OK) return st;
    prof.end(K_CONV3, s);
    prof.begin(K_FC, s);
    st = launch_fc(ws.a3, w.wfc, w.bfc, ws.h, n, g.F, s);
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
    RefWorkspace ws{base, base + f_a1, base + f_a1 + f_a2, base + f_a1 + f_a2 + f_a3};
    float* whead = ws.h + f_h;
    float* bhead = whead + f_wh;
    // every scratch float is written before it is read, so nothing has to start at zero
    HTS_CUDA(cudaMemcpyAsync(whead, w->pi_w, (size_t)g.A * 512 * sizeof(float), cudaMemcpyDeviceToDevice, s));
    HTS_CUDA(cudaMemcpyAsync(whead + (size_t)g.A * 512, w->v_w, 512 * sizeof(float), cudaMemcpyDeviceToDevice, s));
    HTS_CUDA(cudaMemcpyAsync(bhead, w->pi_b, (size_t)g.A * sizeof(float), cudaMemcpyDeviceToDevice, s));
    HTS_CUDA(cudaMemcpyAsync(bhead + g.A, w->v_b, sizeof(float), cudaMemcpyDeviceToDevice, s));
    auto f = [](const void* p) { return const_cast<float*>(static_cast<const float*>(p)); };
    const RefWeights rw{f(w->conv1_w), f(w->conv1_b), f(w->conv2_w), f(w->conv2_b), f(w->conv3_w), f(w->conv3_b),
                        f(w->fc_w), f(w->fc_b), whead, bhead};
    Profiler off;
    hts_status st = ref_forward(g, rw, ws, obs, Indexing{}, nullptr, n, off, s);
    if (st != HTS_OK) return st;
    return launch_heads(ws.h, 1, 0, nullptr, whead, bhead, g.A, env_ids, t_per_env, t, seed, n, Indexing{}, nullptr, actions,
                        logp, values, entropy, logits_or_null, nullptr, s);
}
