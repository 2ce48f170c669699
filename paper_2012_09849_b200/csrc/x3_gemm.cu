// The two tensor-core kernels of the fp32-accurate path (see x3_gemm.cuh for the arithmetic and the layouts).
#include "x3_gemm.cuh"
#include "x3_ring.cuh"
#include "tc_ptx.cuh"
#include "tc_host.cuh"

namespace hts {
using namespace tc;

namespace {

constexpr int kSmemMax = 227 * 1024;
constexpr int kMaxEntries = 4, kMaxStages = 8;

// bf16 operands, fp32 accumulation; `mn_a` / `mn_b`: the operand's tile has its M / N index along the 128-byte rows
__host__ __device__ constexpr uint32_t idesc_x3(uint32_t N, uint32_t mn_a, uint32_t mn_b)
{
    return instr_desc_f16(1, 128, N) | (mn_a << 15) | (mn_b << 16);
}
// Tile with K along the rows (128 bytes of M or N per row, 128-byte swizzle): groups of eight K rows are 1024 bytes
// apart, blocks of 64 M / N elements `lbo_bytes`.
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr, uint32_t lbo_bytes)
{
    return (smem_desc_sw128(addr) & ~((uint64_t)0x3FFF << 16)) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16);
}
__device__ __forceinline__ void tma_load_3d(uint32_t smem_dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(smem_dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void st_v8(void* ptr, const uint32_t* v)
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"l"(ptr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
// One K step of 16: the six products, each weight class into its own accumulator columns [0, NB), [NB, 2 NB), [2 NB, 3 NB).
// With the planes of B stacked along N, plane i of A meets planes 0 .. 2 - i of B in one instruction.
template <int APL, int NB>
__device__ __forceinline__ void mma_x3(uint32_t d, uint64_t a, uint64_t a_plane, uint64_t b, uint32_t mn_a, uint32_t mn_b, bool first)
{
    mma_f16_ss(d, a, b, idesc_x3(3 * NB, 0, 0) | (mn_a << 15) | (mn_b << 16), !first);
    if (APL == 3) {
        mma_f16_ss(d + NB, a + a_plane, b, idesc_x3(2 * NB, 0, 0) | (mn_a << 15) | (mn_b << 16), 1);
        mma_f16_ss(d + 2 * NB, a + 2 * a_plane, b, idesc_x3(NB, 0, 0) | (mn_a << 15) | (mn_b << 16), 1);
    }
}
// Columns [c0, c0 + 32) of an accumulator added to a running sum, its three weight classes smallest first.  WIDE: all
// three in registers at once, one trip to tensor memory instead of two (where the sums leave room for 96 more).
template <int NB, bool WIDE, bool GUARD>
__device__ __forceinline__ void acc_add32(uint32_t taddr, int c0, float* sum)
{
    uint32_t p0[32], p1[32], p2[32], any = 0;
    tmem_ld_32x32(taddr + NB + c0, p1);
    tmem_ld_32x32(taddr + 2 * NB + c0, p2);
    if (WIDE) tmem_ld_32x32(taddr + c0, p0);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 32; ++j) p1[j] = __float_as_uint(__uint_as_float(p1[j]) + __uint_as_float(p2[j]));
    if (!WIDE) {
        tmem_ld_32x32(taddr + c0, p0);
        tmem_ld_wait();
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) any |= p0[j];
    if (GUARD && (any & 0x7f800000u) == 0x7f800000u) {  // none is infinite or NaN otherwise
#pragma unroll
        for (int j = 0; j < 32; ++j) p1[j] = fabsf(__uint_as_float(p0[j])) < INFINITY ? p1[j] : 0;
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) sum[j] += __uint_as_float(p0[j]) + __uint_as_float(p1[j]);
}
// The accumulator is in registers: hand it back.
__device__ __forceinline__ void acc_release(uint64_t* empty_bar, int lane)
{
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(empty_bar);
}

// Persistent: block b takes tiles b, b + blocks, ...  Warp 0 copies (A entries and B stages in two rings), warps 1 and 2
// issue, then eight epilogue warps, two per lane quarter with 32 columns each.  Two accumulators of 192 columns, one for
// each issuing thread, take pairs of B stages (128 of K) in turn; the epilogue adds each to the tile's sum in registers
// (see "Accumulation" in x3_gemm.cuh).
// Bound: shared memory.  An instruction fetches (128 + N) * 32 bytes of operands, 192 clocks per 16 of K (the tensor core
// needs 192, an N of 64 at least 48: 208), and the copies write 4 to 18 KB of A and B meanwhile (30 to 140 clocks): 265 to 310
// clocks are what the issuing threads see (n = 1024, 84 x 84).  So an A entry (all planes, rows 128 + spread) is loaded once
// per tile and every tap reads it shifted, and the weights of an N tile stay in the ring while its M tiles pass, if they
// fit (conv2's 96 KB: gradient of 1024 323 -> 317 us without its forward pass).  One issuing thread: 2 to 3 us more at 5 to 40
// rows, where a tile is a chain of its own, the same at 1024.
// The slots' hand-over is in x3_ring.cuh.
constexpr int kAccs = 2, kThreads = 96 + 256;
struct DgradShared {
    uint64_t a_full[kMaxEntries], a_empty[kMaxEntries], b_full[kMaxStages], b_empty[kMaxStages], d_full[kAccs], d_empty[kAccs];
    uint32_t tmem_slot;
    int abort_flag;
};
// Block `first` of `blocks`.
__device__ __forceinline__ void x3_dgrad(const CUtensorMap& tmA, const CUtensorMap& tmB, const X3TapParams& p, uint8_t* smem_raw, DgradShared& sh,
                                         int first, int blocks)
{
    uint64_t *a_full = sh.a_full, *a_empty = sh.a_empty, *b_full = sh.b_full, *b_empty = sh.b_empty, *d_full = sh.d_full, *d_empty = sh.d_empty;
    volatile int* abortp = &sh.abort_flag;
    constexpr int BB = 3 * 8192;                        // bytes of a B stage: [plane][64 K rows][64 columns]
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int plane_bytes = p.entry_rows * 128;
    const int a_bytes = 3 * plane_bytes, a_pitch = (a_bytes + 1023) & ~1023;
    const uint32_t b_base = base + p.entries * a_pitch;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles = p.m_tiles * p.n_tiles;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kMaxEntries; ++i) { mbar_init(&a_full[i], 1); mbar_init(&a_empty[i], 2); }
        for (int i = 0; i < kMaxStages; ++i) { mbar_init(&b_full[i], 1); mbar_init(&b_empty[i], 2); }
        for (int i = 0; i < kAccs; ++i) { mbar_init(&d_full[i], 1); mbar_init(&d_empty[i], 8); }
        sh.abort_flag = 0;
        fence_barrier_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) tmem_alloc(&sh.tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_d = sh.tmem_slot;
    pdl_wait();
    pdl_trigger();

    const X3Ring ring{p.m_tiles, p.n_tiles, p.chunks, p.taps, p.tpe, p.entries, p.b_stages, first, blocks};
    if (warp == 0) {
        if (lane == 0) {
            struct {
                const CUtensorMap &tmA, &tmB;
                const X3TapParams& p;
                uint64_t *a_full, *a_empty, *b_full, *b_empty;
                volatile int* abortp;
                uint32_t base, b_base;
                int a_bytes, a_pitch;
                __device__ __forceinline__ bool wait_a_empty(int ea, uint32_t par) { return mbar_wait(&a_empty[ea], par, abortp, p.status, 81); }
                __device__ __forceinline__ bool wait_b_empty(int sb, uint32_t par) { return mbar_wait(&b_empty[sb], par, abortp, p.status, 82); }
                __device__ __forceinline__ void load_a(int ea, int mt, int c, int g)
                {
                    mbar_arrive_expect_tx(&a_full[ea], (uint32_t)a_bytes);
                    tma_load_3d(base + ea * a_pitch, &tmA, c * 64, mt * 128 + (p.tpe == 1 ? p.shift[g] : p.lo), 0, &a_full[ea]);
                }
                __device__ __forceinline__ void load_b(int sb, int nt, int c, int tap)
                {
                    mbar_arrive_expect_tx(&b_full[sb], BB);
                    tma_load_3d(b_base + sb * BB, &tmB, tap * p.tap_cols + nt * 64, c * 64, 0, &b_full[sb]);
                }
            } io{tmA, tmB, p, a_full, a_empty, b_full, b_empty, abortp, base, b_base, a_bytes, a_pitch};
            x3_ring_copy(ring, io);
        }
    } else if (warp <= 2) {
        if (lane == 0) {
            const int e = warp - 1;                     // this thread's accumulator: every other accumulation
            struct {
                const X3TapParams& p;
                uint64_t *a_full, *a_empty, *b_full, *b_empty, *d_full, *d_empty;
                volatile int* abortp;
                uint32_t base, b_base, tmem;
                int a_pitch, plane_bytes;
                __device__ __forceinline__ bool wait_a_full(int ea, uint32_t par) { return mbar_wait(&a_full[ea], par, abortp, p.status, 84); }
                __device__ __forceinline__ bool wait_b_full(int sb, uint32_t par) { return mbar_wait(&b_full[sb], par, abortp, p.status, 85); }
                __device__ __forceinline__ bool wait_d_empty(uint32_t par) { return mbar_wait(d_empty, par, abortp, p.status, 83); }
                __device__ __forceinline__ void commit_a_empty(int ea) { mma_commit(&a_empty[ea]); }
                __device__ __forceinline__ void commit_b_empty(int sb) { mma_commit(&b_empty[sb]); }
                __device__ __forceinline__ void commit_d_full() { mma_commit(d_full); }
                __device__ __forceinline__ void arrive_a_empty(int ea) { mbar_arrive(&a_empty[ea]); }
                __device__ __forceinline__ void arrive_b_empty(int sb) { mbar_arrive(&b_empty[sb]); }
                __device__ __forceinline__ void multiply(int ea, int sb, int j, bool start)
                {
                    tc_fence_after();
                    const uint32_t row = p.tpe == 1 ? 0 : (uint32_t)(p.shift[j] - p.lo);
                    const uint64_t a_plane = (uint64_t)(plane_bytes >> 4), a = smem_desc_sw128(base + ea * a_pitch + row * 128);
                    const uint64_t b = smem_desc_mn(b_base + sb * BB, BB / 3);
#pragma unroll
                    for (int k = 0; k < 4; ++k)          // 32 bytes along A's rows, 16 rows of B
                        mma_x3<3, 64>(tmem, a + 2 * k, a_plane, b + 128 * k, 0, 1, start && k == 0);
                }
            } io{p, a_full, a_empty, b_full, b_empty, d_full + e, d_empty + e, abortp, base, b_base, tmem_d + e * 192, a_pitch, plane_bytes};
            x3_ring_issue(ring, e, io);
        }
    } else {
        const int j = (warp - 3) >> 2, q = warp & 3;    // half of the columns; TMEM lane quarter of this warp
        const int row = q * 32 + lane, parts = (p.chunks * p.taps + kX3Part - 1) / kX3Part;
        int it = 0;
        bool alive = true;
        for (int t = first; alive && t < tiles; t += blocks) {
            const int mt = t % p.m_tiles, nt = t / p.m_tiles;
            const int m = mt * 128 + row;
            int env = m / p.P, pix = m - env * p.P;
            int y = pix / p.W, x = pix - y * p.W;
            if (p.mode == X3_DGRAD_FC) { y = nt / p.W_out; x = nt - y * p.W_out; }
            bool ok = env < p.n && y < p.H_out && x < p.W_out;
            size_t off;
            if (p.mode == X3_DGRAD_S2D) {
                const int yy = 2 * y + nt, xx = 2 * x + j;
                ok = env < p.n && yy < p.H_out && xx < p.W_out;
                off = ((size_t)env * p.P_dst + (size_t)yy * p.W_dst + xx) * p.dst_pitch;
            } else
                off = ((size_t)env * p.P_dst + (size_t)y * p.W_dst + x) * p.dst_pitch + j * 32;
            uint32_t mk[16];
            if (ok) {
                const uint4* src = reinterpret_cast<const uint4*>(p.mask + (size_t)m * p.mask_pitch + nt * 64 + j * 32);
#pragma unroll
                for (int i = 0; i < 4; ++i) reinterpret_cast<uint4*>(mk)[i] = src[i];
            }
            float v[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = 0.f;
            for (int s = 0; s < parts; ++s, ++it) {
                const int acc = it % kAccs;
                alive = mbar_wait_warp(&d_full[acc], ((uint32_t)(it / kAccs)) & 1u, abortp, p.status, 86);
                if (!alive) break;
                tc_fence_after();
                acc_add32<64, true, true>(tmem_d + acc * 192 + ((uint32_t)(q * 32) << 16), j * 32, v);
                acc_release(&d_empty[acc], lane);
            }
            if (alive && ok) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {           // positive bf16: sign clear, not zero
                    if ((int16_t)(mk[i] & 0xffffu) <= 0) v[2 * i] = 0.f;
                    if ((int16_t)(mk[i] >> 16) <= 0) v[2 * i + 1] = 0.f;
                }
                __nv_bfloat16* dst = p.dst + off;
#pragma unroll
                for (int h = 0; h < 32; h += 16) {
                    uint32_t o0[8], o1[8], o2[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) x3_split2<true>(v[h + 2 * i], v[h + 2 * i + 1], o0[i], o1[i], o2[i]);
                    st_v8(dst + h, o0);
                    st_v8(dst + p.dst_plane + h, o1);
                    st_v8(dst + 2 * p.dst_plane + h, o2);
                }
            }
            __syncwarp();                               // rows without a destination are here already
        }
    }
    if (*abortp) {                                      // give copies still in flight time to land
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_d, 512);
}
__global__ void __launch_bounds__(kThreads)
x3_dgrad_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const X3TapParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ DgradShared sh;
    x3_dgrad(tmA, tmB, p, smem_raw, sh, blockIdx.x, gridDim.x);
}

// One CTA = (kind, range of row chunks).  Warp 0 copies, warps 1 and 2 issue, two sets of four warps (3..6, 7..10) keep
// the sums in registers (see "Accumulation" in x3_gemm.cuh).  Issuing thread e has accumulators of its own and set e
// adds them up: with two groups it serves group e, with one group every other pair of stages.  An accumulation covers
// 128 rows: two stages of 64, or one of 128 (NB = 32, whose narrow products have two accumulators per thread).  The
// first one of group 0 is a single stage, so that one thread's products run while the other waits for its accumulator
// to be read.  One thread for both groups leaves the tensor core waiting (its instructions come 55 to 70 clocks apart):
// weight gradients of conv3 / conv2 / conv1 / dense at n = 1024, 84 x 84, in launches of their own: 52 / 48 / 43 / 33 us, 43 / 44 / 38 / 30
// with two.
// The sets of kind 0 also sum the columns of B (bias gradient).
// Both operands have the contracted index along their rows (pixels), so tiles go from global memory to the tensor
// core without a transposition; a tap is a row offset into the slab, and the two taps (or slabs) of a group are two
// 64-row blocks of M at a free distance (the leading byte offset).  Tensor core: 208 clocks per 16 rows and group (56 for
// frames); busy for 51 / 54 / 50 % of the time (dense, conv3, conv2 at n = 1024 under ncu, in launches of their own), shared memory
// for as much, DRAM 9 / 19 / 31 %.
constexpr int kWgradThreads = 96 + 256;
struct WgradShared {
    uint64_t full[kMaxStages], empty[kMaxStages], d_full[4], d_empty[4];
    float sum[256][2];
    uint32_t tmem_slot;
    int abort_flag;
};
template <int APL, int NB>
__device__ __forceinline__ void x3_wgrad(const CUtensorMap& tmA, const CUtensorMap& tmB, const X3WgradParams& p, uint8_t* smem_raw, WgradShared& sh,
                                         int block)
{
    constexpr int NACC = NB == 64 ? 2 : 4;              // accumulators
    uint64_t *full = sh.full, *empty = sh.empty, *d_full = sh.d_full, *d_empty = sh.d_empty;
    float (*s_sum)[2] = sh.sum;
    volatile int* abortp = &sh.abort_flag;
    constexpr int BPL = NB == 64 ? 3 : 1;               // NB = 32: the planes are 32-column blocks of one row
    constexpr int ACC = 3 * NB, KR = kX3StageRows<NB>;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
    const int a_slab = (APL * p.a_rows * 128 + 1023) & ~1023, b_plane = KR * 128, b_slab = BPL * b_plane;
    const int a_tx = APL * p.a_rows * 128;
    const int stage_bytes = p.n_a * a_slab + p.n_b * b_slab;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int kind = block / p.ranges;
    if (kind > p.kinds - 1) kind = p.kinds - 1;
    const int range = block - kind * p.ranges;
    const int nr = kind == p.kinds - 1 ? p.last_ranges : p.ranges;
    const int c0 = (int)((long)p.row_chunks * range / nr), c1 = (int)((long)p.row_chunks * (range + 1) / nr);
    const int gi0 = kind * p.group_mul;
    int groups = p.groups;
    if (gi0 + groups > p.group_cap) groups = p.group_cap - gi0;
    const bool biased = p.bias_part && kind == 0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kMaxStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], biased ? 10 : 2); }
        for (int i = 0; i < NACC; ++i) { mbar_init(&d_full[i], 1); mbar_init(&d_empty[i], 4); }
        sh.abort_flag = 0;
        fence_barrier_init();
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) tmem_alloc(&sh.tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_d = sh.tmem_slot;
    pdl_wait();                                         // no trigger: the next kernel's early blocks would crowd a few SMs (1 %)

    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 1;
            const int a_col = (kind % p.ka) * p.a_step, b_col = (kind / p.ka) * p.b_step;
            for (int c = c0; c < c1; ++c) {
                if (!mbar_wait(&empty[s], ph, abortp, p.status, 91)) break;
                mbar_arrive_expect_tx(&full[s], (uint32_t)(p.n_a * a_tx + p.n_b * b_slab));
                const uint32_t dst = base + s * stage_bytes;
                for (int i = 0; i < p.n_a; ++i) {
                    const int k = kind * p.slab_mul + i;
                    tma_load_3d(dst + i * a_slab, &tmA, a_col + p.slab_col[k], c * KR + p.slab_row[k], 0, &full[s]);
                }
                for (int i = 0; i < p.n_b; ++i)
                    tma_load_3d(dst + p.n_a * a_slab + i * b_slab, &tmB, b_col + 64 * i, c * KR, 0, &full[s]);
                if (++s == p.stages) { s = 0; ph ^= 1u; }
            }
        }
    } else if (warp <= 2) {
        if (lane == 0) {
            const int e = warp - 1;
            int s = 0, k = 0;                           // k: accumulation of this thread
            uint32_t ph = 0;
            const uint64_t a_plane = (uint64_t)((p.a_rows * 128) >> 4);
            const uint32_t b_lbo = NB == 64 ? (uint32_t)b_plane : (uint32_t)b_slab;
            const int gi = groups == 2 ? gi0 + e : gi0;
            const uint32_t a_off = (uint32_t)p.a_off[gi], a_lbo = (uint32_t)p.a_lbo[gi], b_off = (uint32_t)(p.n_a * a_slab + p.b_off[gi - gi0]);
            for (int c = c0; c < c1; ++c) {
                const int i = c - c0;
                if (!mbar_wait(&full[s], ph, abortp, p.status, 92)) break;
                if (groups == 2 || ((i >> 1) & 1) == e) {
                    const int half = groups == 2 ? i + 1 - e : i;          // first stage of an accumulation: even
                    const bool first = NB == 32 || i == 0 || (half & 1) == 0;
                    const int acc = NB == 32 ? e + 2 * (k & 1) : e;
                    if (first && !mbar_wait(&d_empty[acc], ((uint32_t)(NB == 32 ? k >> 1 : k) & 1u) ^ 1u, abortp, p.status, 95)) break;
                    tc_fence_after();
                    const uint64_t a = smem_desc_mn(base + s * stage_bytes + a_off, a_lbo);
                    const uint64_t b = smem_desc_mn(base + s * stage_bytes + b_off, b_lbo);
                    const uint32_t d = tmem_d + acc * ACC;
#pragma unroll
                    for (int kk = 0; kk < KR / 16; ++kk)
                        mma_x3<APL, NB>(d, a + 128 * kk, a_plane, b + 128 * kk, 1, 1, first && kk == 0);
                    mma_commit(&empty[s]);
                    if (NB == 32 || (half & 1) == 1 || c == c1 - 1) { mma_commit(&d_full[acc]); ++k; }
                } else
                    mbar_arrive(&empty[s]);
                if (++s == p.stages) { s = 0; ph ^= 1u; }
            }
        }
    } else {
        const int wt = threadIdx.x - 96, set = (warp - 3) >> 2, q = warp & 3, m = q * 32 + lane;
        const uint32_t taddr = tmem_d + ((uint32_t)(q * 32) << 16);
        constexpr int TC = NB / 2;                      // threads along the columns of B (two columns each)
        const int cp = wt % TC, r0 = wt / TC;
        float sum[NB], s0 = 0.f, s1 = 0.f, l0 = 0.f, l1 = 0.f;      // first pieces and lower ones of two columns
#pragma unroll
        for (int j = 0; j < NB; ++j) sum[j] = 0.f;
        bool ok = true;
        int s = 0;
        uint32_t ph = 0;
        int k = 0;                                      // accumulation of this set
        auto drain = [&]() {
            const int acc = NB == 32 ? set + 2 * (k & 1) : set;
            ok = mbar_wait_warp(&d_full[acc], (uint32_t)(NB == 32 ? k >> 1 : k) & 1u, abortp, p.status, 94);
            if (!ok) return;
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < NB; j += 32) acc_add32<NB, NB == 32, APL == 3>(taddr + acc * ACC, j, sum + j);
            acc_release(&d_empty[acc], lane);
            ++k;
        };
        const int n_st = c1 - c0;
        for (int i = 0; ok && i <= n_st; ++i) {         // the columns of stage i, then the accumulations that ended in stage i - 1
            if (biased && i < n_st) {
                ok = mbar_wait_warp(&full[s], ph, abortp, p.status, 93);
                if (!ok) break;
                const uint8_t* b = sm + s * stage_bytes + p.n_a * a_slab;
#pragma unroll 4
                for (int r = r0; r < KR; r += 256 / TC) {
                    uint32_t w[3];
#pragma unroll
                    for (int pl = 0; pl < 3; ++pl) {
                        // byte of the pair inside its 128-byte row, and the row's place (address-based swizzle)
                        const int col = NB == 64 ? cp * 4 : (pl & 1) * 64 + cp * 4;
                        const int blk = NB == 64 ? pl : pl >> 1;
                        const uint32_t off = (uint32_t)(blk * b_plane + r * 128 + (col ^ ((r & 7) << 4)));
                        w[pl] = *reinterpret_cast<const uint32_t*>(b + off);
                    }
                    s0 += __uint_as_float(w[0] << 16); s1 += __uint_as_float(w[0] & 0xffff0000u);
                    l0 += __uint_as_float(w[2] << 16) + __uint_as_float(w[1] << 16);
                    l1 += __uint_as_float(w[2] & 0xffff0000u) + __uint_as_float(w[1] & 0xffff0000u);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
                if (++s == p.stages) { s = 0; ph ^= 1u; }
            }
            const int e = i - 1;
            if (e < 0 || (groups == 1 && ((e >> 1) & 1) != set)) continue;
            if (NB == 32 || ((groups == 2 ? e + 1 - set : e) & 1) || e == n_st - 1) drain();
        }
        if (biased) {
            s_sum[wt][0] = x3_sum(s0, l0); s_sum[wt][1] = x3_sum(s1, l1);
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (wt < NB) {
                float t = 0.f;
                for (int r = 0; r < 256 / TC; ++r) t += s_sum[r * TC + wt / 2][wt & 1];
                p.bias_part[range * NB + wt] = t;
            }
        }
        if (groups == 1) {                              // the stages' buffers are free once both sets are here
            float* other = reinterpret_cast<float*>(sm);
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (set == 1)
#pragma unroll
                for (int j = 0; j < NB; ++j) other[j * 128 + m] = sum[j];
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (set == 0)
#pragma unroll
                for (int j = 0; j < NB; ++j) sum[j] += other[j * 128 + m];
        }
        if (ok && set < groups) {
            const uint32_t* v = reinterpret_cast<const uint32_t*>(sum);
            float* dst = nullptr;
            if (p.fc_w) {
                const int o = (kind % p.ka) * 128 + m, pix = (kind / p.ka) * 2 + set;
                if (pix < p.P3) dst = p.fc_w + (size_t)o * 64 * p.P3 + pix * 64;
            } else
                dst = p.part + (gi0 + set) * p.group_stride + ((size_t)range * 128 + m) * NB;
            if (dst)
#pragma unroll
                for (int i = 0; i < NB; i += 8) st_v8(dst + i, v + i);
        }
    }
    if (*abortp) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem_d, 512);
}

// Two independent passes of the gradient in one launch, each on blocks of its own (one per SM).
__global__ void __launch_bounds__(kWgradThreads)
x3_data_weights_kernel(const __grid_constant__ CUtensorMap dA, const __grid_constant__ CUtensorMap dB, const X3TapParams d, int d_blocks,
                       const __grid_constant__ CUtensorMap wA, const __grid_constant__ CUtensorMap wB, const X3WgradParams w)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ union { DgradShared d; WgradShared w; } sh;
    if ((int)blockIdx.x < d_blocks) x3_dgrad(dA, dB, d, smem_raw, sh.d, blockIdx.x, d_blocks);
    else x3_wgrad<3, 64>(wA, wB, w, smem_raw, sh.w, (int)blockIdx.x - d_blocks);
}
__global__ void __launch_bounds__(kWgradThreads)
x3_weights_kernel(const __grid_constant__ CUtensorMap A2, const __grid_constant__ CUtensorMap B2, const X3WgradParams w2, int blocks2,
                  const __grid_constant__ CUtensorMap A1, const __grid_constant__ CUtensorMap B1, const X3WgradParams w1)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ WgradShared sh;
    if ((int)blockIdx.x < blocks2) x3_wgrad<3, 64>(A2, B2, w2, smem_raw, sh, blockIdx.x);
    else x3_wgrad<1, 32>(A1, B1, w1, smem_raw, sh, (int)blockIdx.x - blocks2);
}
}  // namespace

bool x3_make_map(CUtensorMap* m, const void* ptr, uint64_t cols, uint64_t rows, uint64_t planes, uint64_t pitch_elems,
                 uint64_t plane_elems, uint32_t box_rows, uint32_t box_planes)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {cols, rows, planes};
    const cuuint64_t strides[2] = {pitch_elems * 2, plane_elems * 2};
    const cuuint32_t box[3] = {64, box_rows, box_planes};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool x3_taps_plan(X3TapParams* p, int chunks, int taps, const int* shift)
{
    int lo = shift[0], hi = shift[0];
    for (int i = 0; i < taps; ++i) { lo = shift[i] < lo ? shift[i] : lo; hi = shift[i] > hi ? shift[i] : hi; p->shift[i] = shift[i]; }
    p->taps = taps; p->lo = lo; p->chunks = chunks;
    const int bb = 3 * 8192;
    // every tap reads one A entry shifted; on grids too wide for that (rows of one TMA box, shared memory) each tap
    // loads its own 128 rows
    for (int shared = 1; shared >= 0; --shared) {
        p->tpe = shared ? taps : 1;
        p->entry_rows = shared ? 128 + hi - lo : 128;
        if (p->entry_rows > 256) continue;
        const int a = (3 * p->entry_rows * 128 + 1023) & ~1023;
        p->entries = taps == 1 ? 3 : 2;
        int room = kSmemMax - 4 * 1024 - p->entries * a;
        if (room < 2 * bb) { p->entries = 2; room = kSmemMax - 4 * 1024 - p->entries * a; }
        if (room < 2 * bb) continue;
        p->b_stages = room / bb > kMaxStages ? kMaxStages : room / bb;
        return true;
    }
    return false;
}

namespace {
int dgrad_smem(const X3TapParams& p) { return 1024 + p.entries * ((3 * p.entry_rows * 128 + 1023) & ~1023) + p.b_stages * 3 * 8192; }
template <int APL, int NB>
int wgrad_smem(const X3WgradParams& p)
{
    return 1024 + p.stages * (p.n_a * ((APL * p.a_rows * 128 + 1023) & ~1023) + p.n_b * (NB == 64 ? 3 : 1) * kX3StageRows<NB> * 128);
}
int wgrad_blocks(const X3WgradParams& p) { return p.ranges * (p.kinds - 1) + p.last_ranges; }
constexpr int kRoom = kSmemMax - 3072;                   // the rest is the kernels' static share
}  // namespace

hts_status x3_dgrad_launch(const CUtensorMap& a, const CUtensorMap& b, const X3TapParams& p, cudaStream_t s)
{
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(x3_dgrad_kernel, allowed));
    const int tiles = p.m_tiles * p.n_tiles, sms = device_sm_count(device_slot());
    HTS_CUDA(launch_pdl(x3_dgrad_kernel, dim3(tiles < sms ? tiles : sms), dim3(kThreads), (size_t)dgrad_smem(p), s, a, b, p));
    note_launch();
    return HTS_OK;
}

hts_status x3_data_weights_launch(const CUtensorMap& da, const CUtensorMap& db, const X3TapParams& d, int d_blocks, const CUtensorMap& wa,
                                  const CUtensorMap& wb, const X3WgradParams& w, cudaStream_t s)
{
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(x3_data_weights_kernel, allowed));
    const int sd = dgrad_smem(d), sw = wgrad_smem<3, 64>(w), smem = sd > sw ? sd : sw;
    if (smem > kRoom) return HTS_ERR_SHAPE;
    HTS_CUDA(launch_pdl(x3_data_weights_kernel, dim3(d_blocks + wgrad_blocks(w)), dim3(kWgradThreads), (size_t)smem, s, da, db, d, d_blocks, wa, wb, w));
    note_launch();
    return HTS_OK;
}

hts_status x3_weights_launch(const CUtensorMap& a2, const CUtensorMap& b2, const X3WgradParams& w2, const CUtensorMap& a1, const CUtensorMap& b1,
                             const X3WgradParams& w1, cudaStream_t s)
{
    static OncePerDevice allowed;
    HTS_CUDA(allow_shared(x3_weights_kernel, allowed));
    const int s2 = wgrad_smem<3, 64>(w2), s1 = wgrad_smem<1, 32>(w1), smem = s2 > s1 ? s2 : s1, blocks2 = wgrad_blocks(w2);
    if (smem > kRoom) return HTS_ERR_SHAPE;
    HTS_CUDA(launch_pdl(x3_weights_kernel, dim3(blocks2 + wgrad_blocks(w1)), dim3(kWgradThreads), (size_t)smem, s, a2, b2, w2, blocks2, a1, b1, w1));
    note_launch();
    return HTS_OK;
}

}  // namespace hts
