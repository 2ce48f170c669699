// Shared declarations of the library's translation units (host side + small device helpers).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <atomic>
#include <stdint.h>
#include <utility>
#include "hts.h"

namespace hts {

// ---- launch accounting and error capture --------------------------------------------------
void note_launch(int count = 1);
hts_status cuda_fail(cudaError_t e, const char* where);   // records text, returns HTS_ERR_CUDA
#define HTS_CUDA(call)                                                        \
    do {                                                                      \
        cudaError_t e__ = (call);                                             \
        if (e__ != cudaSuccess) return ::hts::cuda_fail(e__, #call);          \
    } while (0)
#define HTS_LAUNCH_CHECK(name)                                                \
    do {                                                                      \
        ::hts::note_launch();                                                 \
        cudaError_t e__ = cudaGetLastError();                                 \
        if (e__ != cudaSuccess) return ::hts::cuda_fail(e__, name);           \
    } while (0)

// Programmatic dependent launch: the kernel may begin (prologue, weight loads) while its
// predecessor on the stream drains; it must execute pdl_wait() before touching anything the
// predecessor wrote or still reads, and calls pdl_trigger() only after that wait, so that "my
// wait has passed" implies "everything two kernels back is complete" along the whole chain.
// dependent = false: an ordinary launch, for a prologue that reads what the predecessor writes.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(bool dependent, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args)
{
    return launch_chained(true, kernel, grid, block, smem, s, std::forward<Args>(args)...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

inline int conv_out(int extent, int k, int s) { return (extent - k) / s + 1; }

// Kernel attributes (dynamic shared memory, carve-out) belong to a device, and so does the SM count:
// the launchers keep their "already set" marks per device, indexed by this slot.
constexpr int kDeviceSlots = 64;
inline int device_slot()
{
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess) { cudaGetLastError(); d = 0; }
    return (d >= 0 && d < kDeviceSlots) ? d : 0;
}
inline int device_sm_count(int slot)
{
    static int count[kDeviceSlots] = {};
    if (!count[slot]) {
        int d = 0, c = 0;
        if (cudaGetDevice(&d) == cudaSuccess && cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, d) == cudaSuccess) count[slot] = c;
        else cudaGetLastError();
    }
    return count[slot] > 0 ? count[slot] : 1;
}
// Dynamic shared memory and carve-out of a kernel, once per device.  Always as much as the kernel can have: contexts in
// several threads launch it with sizes of their own, and a limit set to one's size could lower what another relies on.
using OncePerDevice = std::atomic<bool>[kDeviceSlots];
template <typename K>
inline cudaError_t allow_shared(K* kernel, OncePerDevice& done, bool carveout = true)
{
    std::atomic<bool>& d = done[device_slot()];
    if (d.load(std::memory_order_acquire)) return cudaSuccess;
    int dev = 0, most = 0;
    cudaFuncAttributes own;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&own, kernel);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)own.sharedSizeBytes);
    if (e == cudaSuccess && carveout) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e == cudaSuccess) d.store(true, std::memory_order_release);
    return e;
}

// Executor-facing addressing of a step (state buffer -> actors -> storage row, Section 4.1): row e of the
// batch reads frame slots[e] of a pool of `pool` frames and writes its outputs at index slots[e].
// slots == nullptr: frames and outputs are dense, row e at index e.  A slot outside [0, pool) is
// reported through the device status word (kStatusBadSlot); that row reads frame 0 and writes nothing.
struct Indexing {
    const int32_t* slots = nullptr;
    int pool = 0;
    int row0 = 0;                      // the batch's rows of the context's workspaces start here
};
constexpr int kStatusBadSlot = 100;
constexpr int kStatusBadAction = 101;     // a stored action outside [0, A) met by the re-evaluation of given actions

// Geometry of the fixed four-layer network for one observation shape.
struct Geometry {
    int C, H, W, A;
    int H1, W1, H2, W2, H3, W3, F;
};

// ---- optional per-kernel event timing of the actor step (benchmark support) ------------------
enum KernelId { K_CONV1 = 0, K_CONV2, K_CONV3, K_FC, K_HEADS, K_COUNT };
struct Profiler {
    static constexpr int kCap = 4096;            // event pairs per kernel between two reads
    bool on = false;
    int used[K_COUNT] = {0, 0, 0, 0, 0};
    cudaEvent_t* start[K_COUNT] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    cudaEvent_t* stop[K_COUNT] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    void begin(int k, cudaStream_t s) { if (on && used[k] < kCap) cudaEventRecord(start[k][used[k]], s); }
    void end(int k, cudaStream_t s) { if (on && used[k] < kCap) { cudaEventRecord(stop[k][used[k]], s); ++used[k]; } }
};

// ---- the fp32 CUDA-core path (the check path for fp32 weights; bf16 contexts never use it) ---
struct RefWeights {            // fp32 device copies in PyTorch layouts
    float *w1, *b1, *w2, *b2, *w3, *b3, *wfc, *bfc;
    float *whead, *bhead;      // [A+1,512], [A+1]: policy rows then the value row
    float *w1k, *w2k, *w3k;    // the convolutions' weights once more as [C k k][O], or nullptr
};
// Rows of one channel: row y is at (y % phases) * phase + (y / phases) * pitch.  A convolution of stride s reads inputs of
// one phase or of s of them.
struct RowLayout { int pitch, phases, phase, chan; };    // one or two phases; the others in elements; chan: between channels
inline RowLayout rows_dense(int H, int W) { return {W, 1, 0, H * W}; }
// Rows of an odd number of 16-byte pieces: eight of them start in eight different sixteenths of the shared-memory banks.
inline RowLayout rows_strips(int H, int W, int phases)
{
    RowLayout l{((W + 3) / 4 | 1) * 4, phases, 0, 0};
    l.phase = (H + phases - 1) / phases * l.pitch; l.chan = phases * l.phase;
    return l;
}
struct RefMaps;                // tensor maps of a context's activations and dense weights (policy_ref.cu)
struct RefWorkspace {          // fp32 activations [n][channels][rows], [n,512]
    float *a1, *a2, *a3, *h;   // a3 is dense
    RowLayout l1, l2;
    const RefMaps* maps;       // or nullptr
    int row0;                  // frame of the maps that is this workspace's first
};
inline RowLayout rows_a1(const Geometry& g) { return rows_strips(g.H1, g.W1, 2); }
inline RowLayout rows_a2(const Geometry& g) { return rows_strips(g.H2, g.W2, 1); }
struct RefPlanes {             // the hidden convolution outputs once more, as three bf16 planes of pixel-major rows
    __nv_bfloat16 *a1, *a2, *a3;
    size_t p1, p2, p3;         // elements between planes
    // Launched behind conv1 if not null: a kernel that needs nothing of it and whose end means conv1's (frames_kernel).
    hts_status (*beside_conv1)(const void* arg, cudaStream_t s);
    const void* arg;
};

// The maps of a workspace for `frames` frames; nullptr if there is no memory or driver for them (its kernels then take other forms).
RefMaps* ref_maps_create(const Geometry& g, const RefWeights& w, const RefWorkspace& ws, size_t frames);
void ref_maps_destroy(RefMaps* maps);
hts_status ref_forward(const Geometry& g, const RefWeights& w, const RefWorkspace& ws,
                       const uint8_t* obs, const Indexing& ix, int* status, int n, Profiler& prof, cudaStream_t s,
                       const RefPlanes* planes = nullptr);
// n frames of activations in rows of a layout as [n][channels][H][W].
hts_status launch_dense_rows(const float* x, const RowLayout& l, int channels, int H, int W, int n, float* out, cudaStream_t s);

// ---- gradient of the learner objective: fp32-accurate passes on the tensor cores (backward.cu) -------
struct X3State;
hts_status x3_create(const Geometry& g, int max_batch, int* status, X3State** out);
void x3_destroy(X3State* t);
// Copies the caller's fp32 weights into the context, and packs them once a gradient has been asked for, in one launch.
hts_status x3_load_weights(X3State* t, const hts_weights& src, const RefWeights& dst, cudaStream_t s);
// The workspace is allocated by the first call on a state.
hts_status x3_gradient(X3State* t, const RefWeights& w, const RefWorkspace& ws, Profiler& prof, const uint8_t* obs, const int32_t* actions, const float* adv, const float* ret,
                       const float* logp_old, float value_coef, float entropy_coef, float clip, int n, const hts_grads& out,
                       bool (*alloc)(void* ctx, void** p, size_t bytes), void* alloc_ctx, cudaStream_t s);

// ---- the tensor-core path (bf16 weights) -------------------------------------------------------
struct TcState;
hts_status tc_check_geometry(const Geometry& g);          // HTS_ERR_SHAPE if the tensor-core kernels cannot take it (no CUDA call)
hts_status tc_create(const Geometry& g, int max_batch, int* status, TcState** out,
                     bool (*alloc)(void* ctx, void** p, size_t bytes), void* alloc_ctx);
void tc_destroy(TcState* t);
hts_status tc_load_weights(TcState* t, const hts_weights& w, cudaStream_t s);
hts_status tc_forward(TcState* t, const uint8_t* obs, const Indexing& ix, int n, Profiler& prof, cudaStream_t s);
hts_status tc_heads(TcState* t, const int32_t* env_ids, const int32_t* t_per_env, int32_t tt, uint64_t seed, int n,
                    const Indexing& ix, int32_t* actions, float* logp, float* values, float* entropy, float* logits,
                    cudaStream_t s, const int32_t* given_actions = nullptr);
hts_status tc_read_activation(TcState* t, int layer, int n, float* out, cudaStream_t s);

// ---- heads + distribution + sampling epilogue (both paths) --------------------------------
// h_partials: [num_splits][n][512] fp32.  If fc_bias != nullptr the hidden vector is
// relu(fc_bias + sum over splits in index order), else it is h_partials[0] as is.
hts_status launch_heads(const float* h_partials, int num_splits, size_t split_stride,
                        const float* fc_bias, const float* whead, const float* bhead, int A,
                        const int32_t* env_ids, const int32_t* t_per_env, int32_t t,
                        uint64_t seed, int n, const Indexing& ix, int* status, int32_t* actions, float* logp,
                        float* values, float* entropy, float* logits, float* h_out, cudaStream_t s,
                        const int32_t* given_actions = nullptr, bool early = true);
// early: a dependent launch may start before this one ends.  given_actions != nullptr: no sampling; row e reports log pi(given_actions[e] | s_e) (env_ids, t and seed are
// not read, actions may be nullptr).  An action outside [0, A) sets kStatusBadAction and the row writes nothing.

hts_status launch_uniforms(const int32_t* env_ids, const int32_t* t_per_env, int32_t t, uint64_t seed, int n,
                           int A, float* out, cudaStream_t s);

// ---- self-test of the bounded wait (reports through the status word like any expired wait) ---
hts_status launch_wait_selftest(long long limit_ticks, int* status, cudaStream_t s);

// ---- advantage scan -------------------------------------------------------------------------
hts_status launch_gae(const float* rewards, const float* values, const uint8_t* dones,
                      const float* bootstrap, float gamma, float lambda, int T, int N,
                      float* adv, float* ret, cudaStream_t s);

// ---- V-trace / truncated importance sampling scan ---------------------------------------------
hts_status launch_vtrace(const float* log_rhos, const float* rewards, const float* values, const uint8_t* dones,
                         const float* bootstrap, float gamma, float lambda, float rho_bar, float c_bar, int T, int N,
                         float* vs, float* pg, cudaStream_t s);

}  // namespace hts
