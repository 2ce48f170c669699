// C ABI of the library: argument validation, context management, launch orchestration.
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include "common.cuh"

namespace hts {

static std::atomic<uint64_t> g_launches{0};
static thread_local char g_cuda_error[256] = "";

void note_launch(int count) { g_launches.fetch_add((uint64_t)count, std::memory_order_relaxed); }

hts_status cuda_fail(cudaError_t e, const char* where)
{
    std::snprintf(g_cuda_error, sizeof(g_cuda_error), "%s: %s", where, cudaGetErrorString(e));
    return HTS_ERR_CUDA;
}

}  // namespace hts

using namespace hts;

struct hts_ctx {
    hts_net_desc desc;
    Geometry g;
    bool loaded = false;
    int last_n = 0;
    RefWeights rw{};              // fp32 check path (weight_dtype fp32)
    RefWorkspace rws{};
    RefMaps* maps = nullptr;
    TcState* tc = nullptr;        // tensor-core path (weight_dtype bf16)
    // staging for the host-buffer entry point: frames, then index words [2][max_batch], result words [4][max_batch] and
    // logits on the device; the words once more in pinned host memory
    uint8_t* s_obs = nullptr;
    int32_t *s_index = nullptr, *s_result = nullptr, *h_words = nullptr;
    float* s_logits = nullptr;
    cudaStream_t h_stream = nullptr;    // its frames' copies, where they are cut in two; null if no batch of the context is
    cudaEvent_t h_start = nullptr, h_copied[2] = {nullptr, nullptr};
    X3State* x3 = nullptr;        // packed weights and workspace of the gradient (weight_dtype fp32)
    int* status = nullptr;        // device status word
    Profiler prof;
    void* allocs[8];
    int nalloc = 0;
};

namespace {

template <typename T>
bool dev_alloc(hts_ctx* c, T** p, size_t count)
{
    void* q = nullptr;
    if (c->nalloc >= 8) return false;
    if (cudaMalloc(&q, count * sizeof(T) + 256) != cudaSuccess) { cudaGetLastError(); return false; }
    c->allocs[c->nalloc++] = q;
    *p = static_cast<T*>(q);
    return true;
}

// Several buffers out of one allocation (an allocation costs tens of microseconds; a context has some thirty buffers).
struct Carve {
    struct Item { void** p; size_t bytes; } items[40];
    int n = 0;
    size_t total = 0;
    template <typename T>
    void add(T** p, size_t count)
    {
        items[n++] = {reinterpret_cast<void**>(p), total};
        total += (count * sizeof(T) + 256 + 255) & ~(size_t)255;
    }
    bool alloc(hts_ctx* c)
    {
        uint8_t* base = nullptr;
        if (!dev_alloc(c, &base, total)) return false;
        for (int i = 0; i < n; ++i) *items[i].p = base + items[i].bytes;
        return true;
    }
};

bool raw_alloc(void* c, void** p, size_t bytes)
{
    uint8_t* q = nullptr;
    if (!dev_alloc(static_cast<hts_ctx*>(c), &q, bytes)) return false;
    *p = q;
    return true;
}

struct Range { const void* p; size_t bytes; };
bool overlaps(const Range& a, const Range& b)
{
    if (!a.p || !b.p || !a.bytes || !b.bytes) return false;
    const uintptr_t a0 = (uintptr_t)a.p, a1 = a0 + a.bytes, b0 = (uintptr_t)b.p, b1 = b0 + b.bytes;
    return a0 < b1 && b0 < a1;
}
// outputs must not overlap inputs or each other
bool any_overlap(const Range* in, int nin, const Range* out, int nout)
{
    for (int i = 0; i < nout; ++i) {
        for (int j = 0; j < nin; ++j) if (overlaps(out[i], in[j])) return true;
        for (int j = i + 1; j < nout; ++j) if (overlaps(out[i], out[j])) return true;
    }
    return false;
}

hts_status check_step_args(hts_ctx* ctx, const void* obs, const void* env_ids, int n,
                           const void* actions, const void* logp, const void* values, const void* entropy,
                           bool on_host = false)
{
    if (!ctx || !obs || !env_ids || !actions || !logp || !values || !entropy) return HTS_ERR_INVALID_ARG;
    if (n < 1 || n > ctx->desc.max_batch) return HTS_ERR_INVALID_ARG;
    // the tensor-core path stages frames with bulk copies, which need 16-byte-aligned global addresses
    // (frame, channel and row-group offsets are multiples of 16 because H and W are multiples of 4)
    if (ctx->tc && !on_host && ((uintptr_t)obs & 15u) != 0) return HTS_ERR_INVALID_ARG;
    if (!ctx->loaded) return HTS_ERR_UNSUPPORTED;
    return HTS_OK;
}

hts_status run_step(hts_ctx* ctx, const uint8_t* obs, const Indexing& ix, const int32_t* env_ids, const int32_t* t_per_env,
                    int32_t t, uint64_t seed, int32_t n, int32_t* actions, float* logp, float* values,
                    float* entropy, float* logits, cudaStream_t s, const int32_t* given_actions = nullptr)
{
    const Geometry& g = ctx->g;
    hts_status st;
    if (ctx->tc) {
        st = tc_forward(ctx->tc, obs, ix, n, ctx->prof, s);
        if (st != HTS_OK) return st;
        ctx->prof.begin(K_HEADS, s);
        st = tc_heads(ctx->tc, env_ids, t_per_env, t, seed, n, ix, actions, logp, values, entropy, logits, s, given_actions);
    } else {
        const size_t r = (size_t)ix.row0;
        RefWorkspace ws = ctx->rws;
        ws.row0 = ix.row0; ws.a1 += r * 32 * ws.l1.chan; ws.a2 += r * 64 * ws.l2.chan; ws.a3 += r * g.F; ws.h += r * 512;
        st = ref_forward(g, ctx->rw, ws, obs, ix, ctx->status, n, ctx->prof, s);
        if (st != HTS_OK) return st;
        ctx->prof.begin(K_HEADS, s);
        st = launch_heads(ws.h, 1, 0, nullptr, ctx->rw.whead, ctx->rw.bhead, g.A, env_ids, t_per_env, t,
                          seed, n, ix, ctx->status, actions, logp, values, entropy, logits, nullptr, s, given_actions, false);
    }
    if (st != HTS_OK) return st;
    ctx->prof.end(K_HEADS, s);
    ctx->last_n = ix.row0 + n;
    return HTS_OK;
}

}  // namespace

// Rows up to which the kernels use the context's pinned words directly.  Call with the words / with copies, us: 37.0 / 46.0 (1 row),
// 55.4 / 58.4 (32), 108.6 / 114.5 (128), 149.0 / 153.7 (192), 320.7 / 330.2 (512), 601 / 609 (1024), 1165 / 1169 (2048),
// 2265 / 2258 (4096), 4484 / 4461 (8192): the two cross between 2048 and 4096 rows, so the line could lie higher.
constexpr int kHostDirect = 128;

// The frames of a host step are copied in two parts, so that the step of the first runs while the second is copied.  It pays if
// the second part's copy outlasts the first part's step, and if what then remains, the second part's step, is shorter than the
// whole one by more than another copy and chain of launches cost.
// bf16: a step of n rows takes 16 to 20 us and a sixteenth (60 x 60) to a forty-fifth (72 x 96, 16 channels) of what the n frames'
// copy takes (55 bytes per ns), so the second part is 2 MB and an eighteenth of all bytes.  Host step with second parts of fewer rows /
// about as many / more, us: 1024 of 84 x 84 x 4 593.8 (48 rows) / 575 (96 to 128) / 577.6 (144); 512 of 72 x 96 x 16 1082.1 (16) / 1079.6
// (48) / 1082.3 (128); 512 of 84 x 84 x 8 579.7 (32) / 577.6 (64) / 579.2 (128); 2048 of 36 x 44 299.3 (128) / 287.7 (448) / 291.4 (640).
// Small frames' steps save less than their share of the bytes: the line is 5.2 MB and 4 KB for each row.  One part / two, us:
//   36 x 44 x 4   6 MB 158.9 / 164.8   7 MB 177.5 / 187.1   10 MB 236.4 / 236.0   14 MB 315.3 / 315.2   20 MB 433.2 / 427.5   51 MB 1021 / 993
//   60 x 60 x 4   6 MB 158.3 / 161.4   7 MB 176.5 / 181.8   8 MB 201.4 / 198.5    12 MB 274.3 / 273.6   16 MB 354.8 / 339.5   40 MB 810 / 780
//   64 x 96 x 4   6.3 MB 165.8 / 162.8   8 MB 198.5 / 194.0   12 MB 274.1 / 265.3   24 MB 502.5 / 487.9
//   84 x 84 x 4   7.2 MB 182.6 / 181.9   8 MB 197.8 / 193.9   12 MB 273.1 / 266.6   28.9 MB 595.9 / 575.7   57.8 MB 1141 / 1104
//   84 x 84 x 8   14.5 MB 316.8 / 314.3   29 MB 584.7 / 578.2   57 MB 1107 / 1086
//   72 x 96 x 16   28.4 MB 570.7 / 567.0   57 MB 1097 / 1086   110 MB 2071 / 2042
// and 256 rows: below two per SM the step is one observation's latency, whatever it is cut into (159 of 84 x 84 x 8 216.0 / 216.3, 124
// of them 174.9 / 186.4; 144 of 72 x 96 x 16 343.1 / 342.7).
// fp32 steps take as long as their copies: halves, from 512 rows.  513 of 84 x 84 x 4 618.8 / 557.1, 631 of 36 x 44 191.4 / 183.3 (394 of
// them 139.3 / 144.8), 515 of 72 x 96 x 16 1567 / 1346.
namespace {
int host_first_rows(const hts_ctx* ctx, int n)
{
    if (!ctx->tc) return n >= 512 ? n / 2 : n;
    const long long frame = (long long)ctx->g.C * ctx->g.H * ctx->g.W, bytes = n * frame;
    if (n < 256 || bytes < 5200000 + 4000LL * n) return n;
    return n - (int)((2000000 + bytes / 18 + frame - 1) / frame);
}
// Stream and events of the copies.  A stream takes 56 to 66 us to make, more than a cut saves: it is made with the context, if the
// context's largest batch is cut.  Without them frames are copied in one part.
void make_host_copies(hts_ctx* c)
{
    if (host_first_rows(c, c->desc.max_batch) == c->desc.max_batch) return;
    bool ok = true;
    for (cudaEvent_t* e : {&c->h_start, &c->h_copied[0], &c->h_copied[1]}) ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
    if (!ok || cudaStreamCreateWithFlags(&c->h_stream, cudaStreamNonBlocking) != cudaSuccess) {
        c->h_stream = nullptr;
        cudaGetLastError();
    }
}
}  // namespace

// staging buffer of hts_gae_host, one per device; grows on demand, freed by hts_gae_host_release
static char* g_gae_stage[kDeviceSlots] = {};
static size_t g_gae_stage_bytes[kDeviceSlots] = {};

extern "C" {

hts_status hts_policy_create(const hts_net_desc* d, hts_ctx** out)
{
    if (!d || !out) return HTS_ERR_INVALID_ARG;
    *out = nullptr;
    if (d->C < 1 || d->H < 1 || d->W < 1 || d->max_batch < 1) return HTS_ERR_INVALID_ARG;
    if (d->num_actions < 1 || d->num_actions > 64) return HTS_ERR_INVALID_ARG;
    if (d->weight_dtype != HTS_DTYPE_FP32 && d->weight_dtype != HTS_DTYPE_BF16) return HTS_ERR_INVALID_ARG;
    if (d->H % 4 || d->W % 4 || d->C > 64) return HTS_ERR_SHAPE;
    Geometry g{};
    g.C = d->C; g.H = d->H; g.W = d->W; g.A = d->num_actions;
    if (g.H < 8 || g.W < 8) return HTS_ERR_SHAPE;
    g.H1 = conv_out(g.H, 8, 4); g.W1 = conv_out(g.W, 8, 4);
    if (g.H1 < 4 || g.W1 < 4) return HTS_ERR_SHAPE;
    g.H2 = conv_out(g.H1, 4, 2); g.W2 = conv_out(g.W1, 4, 2);
    if (g.H2 < 3 || g.W2 < 3) return HTS_ERR_SHAPE;
    g.H3 = conv_out(g.H2, 3, 1); g.W3 = conv_out(g.W2, 3, 1);
    g.F = 64 * g.H3 * g.W3;
    if (d->weight_dtype == HTS_DTYPE_BF16) {                 // shape limits of the tensor-core kernels, before any CUDA call
        const hts_status gs = tc_check_geometry(g);
        if (gs != HTS_OK) return gs;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cuda_fail(cudaGetLastError(), "cudaGetDevice");

    hts_ctx* c = new (std::nothrow) hts_ctx();
    if (!c) return HTS_ERR_ALLOC;
    c->desc = *d; c->g = g;
    const size_t nb = (size_t)d->max_batch;
    const int A = g.A;
    Carve cv;
    cv.add(&c->status, 1);
    cv.add(&c->s_obs, nb * g.C * g.H * g.W);
    cv.add(&c->s_index, 2 * nb); cv.add(&c->s_result, 4 * nb); cv.add(&c->s_logits, nb * A);
    if (d->weight_dtype == HTS_DTYPE_FP32) {
        cv.add(&c->rw.w1, (size_t)32 * g.C * 64); cv.add(&c->rw.b1, 32);
        cv.add(&c->rw.w2, (size_t)64 * 32 * 16); cv.add(&c->rw.b2, 64);
        cv.add(&c->rw.w3, (size_t)64 * 64 * 9); cv.add(&c->rw.b3, 64);
        cv.add(&c->rw.wfc, (size_t)512 * g.F); cv.add(&c->rw.bfc, 512);
        cv.add(&c->rw.whead, (size_t)(A + 1) * 512); cv.add(&c->rw.bhead, (size_t)A + 1);
        cv.add(&c->rw.w1k, (size_t)32 * g.C * 64); cv.add(&c->rw.w2k, (size_t)64 * 32 * 16); cv.add(&c->rw.w3k, (size_t)64 * 64 * 9);
        c->rws.l1 = rows_a1(g); c->rws.l2 = rows_a2(g);
        cv.add(&c->rws.a1, nb * 32 * c->rws.l1.chan); cv.add(&c->rws.a2, nb * 64 * c->rws.l2.chan);
        cv.add(&c->rws.a3, nb * g.F); cv.add(&c->rws.h, nb * 512);
    }
    if (!cv.alloc(c)) { hts_policy_destroy(c); return HTS_ERR_ALLOC; }
    const hts_status st = d->weight_dtype == HTS_DTYPE_BF16 ? tc_create(g, d->max_batch, c->status, &c->tc, raw_alloc, c)
                                                            : x3_create(g, d->max_batch, c->status, &c->x3);
    if (st != HTS_OK) { hts_policy_destroy(c); return st; }
    if (!c->tc) c->rws.maps = c->maps = ref_maps_create(g, c->rw, c->rws, nb);
    if (cudaMemset(c->status, 0, sizeof(int)) != cudaSuccess) {
        hts_status st = cuda_fail(cudaGetLastError(), "cudaMemset");
        hts_policy_destroy(c);
        return st;
    }
    make_host_copies(c);
    *out = c;
    return HTS_OK;
}

hts_status hts_policy_load_weights(hts_ctx* ctx, const hts_weights* w, void* cuda_stream)
{
    if (!ctx || !w) return HTS_ERR_INVALID_ARG;
    const void* const* p = reinterpret_cast<const void* const*>(w);
    for (int i = 0; i < 12; ++i) if (!p[i]) return HTS_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const hts_status st = ctx->tc ? tc_load_weights(ctx->tc, *w, s) : x3_load_weights(ctx->x3, *w, ctx->rw, s);
    if (st != HTS_OK) return st;
    ctx->loaded = true;
    return HTS_OK;
}

hts_status hts_policy_step(hts_ctx* ctx, const uint8_t* obs, const int32_t* env_ids,
                           const int32_t* t_per_env, int32_t t, uint64_t seed, int32_t n,
                           int32_t* actions, float* logp, float* values, float* entropy,
                           float* logits_or_null, void* cuda_stream)
{
    hts_status st = check_step_args(ctx, obs, env_ids, n, actions, logp, values, entropy);
    if (st != HTS_OK) return st;
    const size_t nn = (size_t)n;
    const Range in[] = {{obs, nn * ctx->g.C * ctx->g.H * ctx->g.W}, {env_ids, nn * 4}, {t_per_env, nn * 4}};
    const Range outr[] = {{actions, nn * 4}, {logp, nn * 4}, {values, nn * 4}, {entropy, nn * 4},
                          {logits_or_null, nn * ctx->g.A * 4}};
    if (any_overlap(in, 3, outr, 5)) return HTS_ERR_INVALID_ARG;
    return run_step(ctx, obs, Indexing{}, env_ids, t_per_env, t, seed, n, actions, logp, values, entropy, logits_or_null,
                    static_cast<cudaStream_t>(cuda_stream));
}

hts_status hts_policy_step_indexed(hts_ctx* ctx, const uint8_t* state_buffer, int32_t pool, const int32_t* slots,
                                   const int32_t* env_ids, const int32_t* t_per_env, int32_t t, uint64_t seed,
                                   int32_t n, int32_t* actions_row, float* logp_row, float* values_row,
                                   float* entropy_row, void* cuda_stream)
{
    hts_status st = check_step_args(ctx, state_buffer, env_ids, n, actions_row, logp_row, values_row, entropy_row);
    if (st != HTS_OK) return st;
    if (!slots || pool < 1) return HTS_ERR_INVALID_ARG;
    const size_t nn = (size_t)n, pp = (size_t)pool;
    const Range in[] = {{state_buffer, pp * ctx->g.C * ctx->g.H * ctx->g.W}, {slots, nn * 4}, {env_ids, nn * 4},
                        {t_per_env, nn * 4}};
    const Range outr[] = {{actions_row, pp * 4}, {logp_row, pp * 4}, {values_row, pp * 4}, {entropy_row, pp * 4}};
    if (any_overlap(in, 4, outr, 4)) return HTS_ERR_INVALID_ARG;
    Indexing ix;
    ix.slots = slots; ix.pool = pool;
    return run_step(ctx, state_buffer, ix, env_ids, t_per_env, t, seed, n, actions_row, logp_row, values_row, entropy_row,
                    nullptr, static_cast<cudaStream_t>(cuda_stream));
}

hts_status hts_policy_evaluate(hts_ctx* ctx, const uint8_t* obs, const int32_t* actions, int32_t n, float* logp,
                               float* values, float* entropy, float* logits_or_null, void* cuda_stream)
{
    if (!ctx || !obs || !actions || !logp || !values || !entropy) return HTS_ERR_INVALID_ARG;
    if (n < 1 || n > ctx->desc.max_batch) return HTS_ERR_INVALID_ARG;
    if (ctx->tc && ((uintptr_t)obs & 15u) != 0) return HTS_ERR_INVALID_ARG;
    if (!ctx->loaded) return HTS_ERR_UNSUPPORTED;
    const size_t nn = (size_t)n;
    const Range in[] = {{obs, nn * ctx->g.C * ctx->g.H * ctx->g.W}, {actions, nn * 4}};
    const Range outr[] = {{logp, nn * 4}, {values, nn * 4}, {entropy, nn * 4}, {logits_or_null, nn * ctx->g.A * 4}};
    if (any_overlap(in, 2, outr, 4)) return HTS_ERR_INVALID_ARG;
    return run_step(ctx, obs, Indexing{}, nullptr, nullptr, 0, 0, n, nullptr, logp, values, entropy, logits_or_null,
                    static_cast<cudaStream_t>(cuda_stream), actions);
}

hts_status hts_policy_gradient(hts_ctx* ctx, const uint8_t* obs, const int32_t* actions, const float* advantages,
                               const float* returns, const float* logp_old_or_null, float value_coef, float entropy_coef,
                               float clip, int32_t n, const hts_grads* grads, void* cuda_stream)
{
    if (!ctx || !obs || !actions || !advantages || !returns || !grads) return HTS_ERR_INVALID_ARG;
    float* const* gp = reinterpret_cast<float* const*>(grads);
    for (int i = 0; i < 12; ++i) if (!gp[i]) return HTS_ERR_INVALID_ARG;
    if (n < 1 || n > ctx->desc.max_batch) return HTS_ERR_INVALID_ARG;
    if (!(clip >= 0.f) || !std::isfinite(clip) || !std::isfinite(value_coef) || !std::isfinite(entropy_coef)) return HTS_ERR_INVALID_ARG;
    if (ctx->tc) return HTS_ERR_UNSUPPORTED;
    if (!ctx->loaded) return HTS_ERR_UNSUPPORTED;
    const hts_status st = x3_gradient(ctx->x3, ctx->rw, ctx->rws, ctx->prof, obs, actions, advantages, returns, logp_old_or_null,
                                      value_coef, entropy_coef, clip, n, *grads, raw_alloc, ctx, static_cast<cudaStream_t>(cuda_stream));
    if (st == HTS_OK) ctx->last_n = n;
    return st;
}

hts_status hts_policy_step_host(hts_ctx* ctx, const uint8_t* obs, const int32_t* env_ids,
                                const int32_t* t_per_env, int32_t t, uint64_t seed, int32_t n,
                                int32_t* actions, float* logp, float* values, float* entropy,
                                float* logits_or_null, void* cuda_stream)
{
    hts_status st = check_step_args(ctx, obs, env_ids, n, actions, logp, values, entropy, true);
    if (st != HTS_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const size_t nn = (size_t)n, nb = (size_t)ctx->desc.max_batch;
    // A copy costs about 4 us of the host and 2 of the stream whatever it carries, so the index and result words of a
    // call pass through the context's pinned words: small batches' kernels read and write those themselves, larger ones
    // take one copy each way (the heads kernel's 4-byte accesses each cross the bus).
    if (!ctx->h_words && cudaHostAlloc(reinterpret_cast<void**>(&ctx->h_words), 6 * nb * 4, cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        return HTS_ERR_ALLOC;
    }
    int32_t *h_in = ctx->h_words, *h_out = ctx->h_words + 2 * nb;
    std::memcpy(h_in, env_ids, nn * 4);
    if (t_per_env) std::memcpy(h_in + nn, t_per_env, nn * 4);
    const bool direct = n <= kHostDirect;
    int32_t *in = direct ? h_in : ctx->s_index, *out = direct ? h_out : ctx->s_result;
    if (!direct) HTS_CUDA(cudaMemcpyAsync(in, h_in, (t_per_env ? 2 : 1) * nn * 4, cudaMemcpyHostToDevice, s));
    float* outf = reinterpret_cast<float*>(out);
    const size_t frame = (size_t)ctx->g.C * ctx->g.H * ctx->g.W;
    auto step = [&](int row0, int rows) {
        Indexing ix;
        ix.row0 = row0;
        return run_step(ctx, ctx->s_obs + row0 * frame, ix, in + row0, t_per_env ? in + nn + row0 : nullptr, t, seed, rows, out + row0,
                        outf + nn + row0, outf + 2 * nn + row0, outf + 3 * nn + row0,
                        logits_or_null ? ctx->s_logits + (size_t)row0 * ctx->g.A : nullptr, s);
    };
    const int first = host_first_rows(ctx, n);
    if (first < n && ctx->h_stream) {
        HTS_CUDA(cudaEventRecord(ctx->h_start, s));        // what the stream still does to the caller's frames comes first
        HTS_CUDA(cudaStreamWaitEvent(ctx->h_stream, ctx->h_start, 0));
        cudaError_t e = cudaSuccess;
        for (int part = 0; part < 2 && st == HTS_OK && e == cudaSuccess; ++part) {
            const int row0 = part ? first : 0, rows = part ? n - first : first;
            e = cudaMemcpyAsync(ctx->s_obs + row0 * frame, obs + row0 * frame, rows * frame, cudaMemcpyHostToDevice, ctx->h_stream);
            if (e == cudaSuccess) e = cudaEventRecord(ctx->h_copied[part], ctx->h_stream);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ctx->h_copied[part], 0);
            if (e == cudaSuccess) st = step(row0, rows);
        }
        if (st != HTS_OK || e != cudaSuccess) {
            cudaStreamSynchronize(ctx->h_stream);          // the caller's buffer is free again
            return st != HTS_OK ? st : cuda_fail(e, "hts_policy_step_host");
        }
    } else {
        HTS_CUDA(cudaMemcpyAsync(ctx->s_obs, obs, nn * frame, cudaMemcpyHostToDevice, s));
        st = step(0, n);
        if (st != HTS_OK) return st;
    }
    if (!direct) HTS_CUDA(cudaMemcpyAsync(h_out, out, 4 * nn * 4, cudaMemcpyDeviceToHost, s));
    if (logits_or_null)
        HTS_CUDA(cudaMemcpyAsync(logits_or_null, ctx->s_logits, nn * ctx->g.A * 4, cudaMemcpyDeviceToHost, s));
    HTS_CUDA(cudaStreamSynchronize(s));
    std::memcpy(actions, h_out, nn * 4);
    std::memcpy(logp, h_out + nn, nn * 4);
    std::memcpy(values, h_out + 2 * nn, nn * 4);
    std::memcpy(entropy, h_out + 3 * nn, nn * 4);
    return HTS_OK;
}

hts_status hts_policy_read_activation(hts_ctx* ctx, int32_t layer, int32_t n, float* out, void* cuda_stream)
{
    if (!ctx || !out || layer < 1 || layer > 4) return HTS_ERR_INVALID_ARG;
    if (n < 1 || n > ctx->last_n) return HTS_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    if (ctx->tc) return tc_read_activation(ctx->tc, layer, n, out, s);
    const Geometry& g = ctx->g;
    if (layer == 1) return launch_dense_rows(ctx->rws.a1, ctx->rws.l1, 32, g.H1, g.W1, n, out, s);
    if (layer == 2) return launch_dense_rows(ctx->rws.a2, ctx->rws.l2, 64, g.H2, g.W2, n, out, s);
    const float* src = layer == 3 ? ctx->rws.a3 : ctx->rws.h;
    const size_t per = layer == 3 ? (size_t)g.F : 512;
    HTS_CUDA(cudaMemcpyAsync(out, src, per * n * sizeof(float), cudaMemcpyDeviceToDevice, s));
    return HTS_OK;
}

hts_status hts_action_uniforms(const int32_t* env_ids, const int32_t* t_per_env, int32_t t, uint64_t seed,
                               int32_t n, int32_t num_actions, float* out, void* cuda_stream)
{
    if (!env_ids || !out || n < 1 || num_actions < 1 || num_actions > 64) return HTS_ERR_INVALID_ARG;
    return launch_uniforms(env_ids, t_per_env, t, seed, n, num_actions, out, static_cast<cudaStream_t>(cuda_stream));
}

hts_status hts_last_async_error(hts_ctx* ctx)
{
    if (!ctx) return HTS_ERR_INVALID_ARG;
    int word = 0;
    HTS_CUDA(cudaMemcpy(&word, ctx->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (word != 0) {
        HTS_CUDA(cudaMemset(ctx->status, 0, sizeof(int)));
        return (word == kStatusBadSlot || word == kStatusBadAction) ? HTS_ERR_INVALID_ARG : HTS_ERR_TIMEOUT;
    }
    return HTS_OK;
}

hts_status hts_wait_selftest(hts_ctx* ctx, int64_t limit_ticks, void* cuda_stream)
{
    if (!ctx || limit_ticks < 1000 || limit_ticks > 100000000LL) return HTS_ERR_INVALID_ARG;
    return launch_wait_selftest((long long)limit_ticks, ctx->status, static_cast<cudaStream_t>(cuda_stream));
}

hts_status hts_policy_profile(hts_ctx* ctx, int32_t enable)
{
    if (!ctx) return HTS_ERR_INVALID_ARG;
    Profiler& p = ctx->prof;
    if (enable && !p.start[0]) {
        for (int k = 0; k < K_COUNT; ++k) {
            p.start[k] = new (std::nothrow) cudaEvent_t[Profiler::kCap]();
            p.stop[k] = new (std::nothrow) cudaEvent_t[Profiler::kCap]();
            if (!p.start[k] || !p.stop[k]) return HTS_ERR_ALLOC;
            for (int i = 0; i < Profiler::kCap; ++i) {
                HTS_CUDA(cudaEventCreate(&p.start[k][i]));
                HTS_CUDA(cudaEventCreate(&p.stop[k][i]));
            }
        }
    }
    if (enable) for (int k = 0; k < K_COUNT; ++k) p.used[k] = 0;
    p.on = enable != 0;
    return HTS_OK;
}

hts_status hts_policy_profile_read(hts_ctx* ctx, int32_t kernel, float* total_ms, int32_t* launches)
{
    if (!ctx || !total_ms || !launches || kernel < 0 || kernel >= K_COUNT) return HTS_ERR_INVALID_ARG;
    Profiler& p = ctx->prof;
    float sum = 0.f;
    for (int i = 0; i < p.used[kernel]; ++i) {
        float ms = 0.f;
        HTS_CUDA(cudaEventSynchronize(p.stop[kernel][i]));
        HTS_CUDA(cudaEventElapsedTime(&ms, p.start[kernel][i], p.stop[kernel][i]));
        sum += ms;
    }
    *total_ms = sum;
    *launches = p.used[kernel];
    return HTS_OK;
}

const char* hts_policy_kernel_name(int32_t kernel)
{
    static const char* names[K_COUNT] = {"conv1", "conv2", "conv3", "fc", "heads"};
    return (kernel >= 0 && kernel < K_COUNT) ? names[kernel] : "";
}

void hts_policy_destroy(hts_ctx* ctx)
{
    if (!ctx) return;
    for (int k = 0; k < K_COUNT; ++k) {
        if (ctx->prof.start[k]) { for (int i = 0; i < Profiler::kCap; ++i) cudaEventDestroy(ctx->prof.start[k][i]); delete[] ctx->prof.start[k]; }
        if (ctx->prof.stop[k]) { for (int i = 0; i < Profiler::kCap; ++i) cudaEventDestroy(ctx->prof.stop[k][i]); delete[] ctx->prof.stop[k]; }
    }
    if (ctx->tc) tc_destroy(ctx->tc);
    if (ctx->x3) x3_destroy(ctx->x3);
    if (ctx->maps) ref_maps_destroy(ctx->maps);
    for (int i = 0; i < ctx->nalloc; ++i) cudaFree(ctx->allocs[i]);
    if (ctx->h_words) cudaFreeHost(ctx->h_words);
    for (cudaEvent_t e : {ctx->h_start, ctx->h_copied[0], ctx->h_copied[1]}) if (e) cudaEventDestroy(e);
    if (ctx->h_stream) cudaStreamDestroy(ctx->h_stream);
    delete ctx;
}

static hts_status check_gae_args(const void* r, const void* v, const void* d, const void* b, float gamma,
                                 float lambda, int T, int N, const void* adv, const void* ret)
{
    if (!r || !v || !d || !b || !adv || !ret) return HTS_ERR_INVALID_ARG;
    if (T < 1 || N < 1) return HTS_ERR_INVALID_ARG;
    if (!(gamma >= 0.f && gamma <= 1.f) || !(lambda >= 0.f && lambda <= 1.f)) return HTS_ERR_INVALID_ARG;   // NaN fails both
    return HTS_OK;
}

hts_status hts_gae(const float* rewards, const float* values, const uint8_t* dones, const float* bootstrap,
                   float gamma, float lambda, int32_t T, int32_t N, float* advantages, float* returns,
                   void* cuda_stream)
{
    hts_status st = check_gae_args(rewards, values, dones, bootstrap, gamma, lambda, T, N, advantages, returns);
    if (st != HTS_OK) return st;
    const size_t tn = (size_t)T * N;
    const Range in[] = {{rewards, tn * 4}, {values, tn * 4}, {dones, tn}, {bootstrap, (size_t)N * 4}};
    const Range outr[] = {{advantages, tn * 4}, {returns, tn * 4}};
    if (any_overlap(in, 4, outr, 2)) return HTS_ERR_INVALID_ARG;
    return launch_gae(rewards, values, dones, bootstrap, gamma, lambda, T, N, advantages, returns,
                      static_cast<cudaStream_t>(cuda_stream));
}

hts_status hts_vtrace(const float* log_rhos, const float* rewards, const float* values, const uint8_t* dones,
                      const float* bootstrap, float gamma, float lambda, float rho_bar, float c_bar, int32_t T, int32_t N,
                      float* vs, float* pg_advantages, void* cuda_stream)
{
    hts_status st = check_gae_args(rewards, values, dones, bootstrap, gamma, lambda, T, N, vs, pg_advantages);
    if (st != HTS_OK) return st;
    if (!log_rhos || !(rho_bar >= 0.f) || !(c_bar >= 0.f)) return HTS_ERR_INVALID_ARG;      // NaN fails both
    const size_t tn = (size_t)T * N;
    const Range in[] = {{log_rhos, tn * 4}, {rewards, tn * 4}, {values, tn * 4}, {dones, tn}, {bootstrap, (size_t)N * 4}};
    const Range outr[] = {{vs, tn * 4}, {pg_advantages, tn * 4}};
    if (any_overlap(in, 5, outr, 2)) return HTS_ERR_INVALID_ARG;
    return launch_vtrace(log_rhos, rewards, values, dones, bootstrap, gamma, lambda, rho_bar, c_bar, T, N, vs, pg_advantages,
                         static_cast<cudaStream_t>(cuda_stream));
}

hts_status hts_gae_host(const float* rewards, const float* values, const uint8_t* dones, const float* bootstrap,
                        float gamma, float lambda, int32_t T, int32_t N, float* advantages, float* returns,
                        void* cuda_stream)
{
    hts_status st = check_gae_args(rewards, values, dones, bootstrap, gamma, lambda, T, N, advantages, returns);
    if (st != HTS_OK) return st;
    const int dev = device_slot();
    char*& stage = g_gae_stage[dev];
    size_t& stage_bytes = g_gae_stage_bytes[dev];
    const size_t tn = (size_t)T * N;
    const size_t tn4 = (tn * 4 + 255) / 256 * 256, tn1 = (tn + 255) / 256 * 256, n4 = ((size_t)N * 4 + 255) / 256 * 256;
    const size_t need = 4 * tn4 + tn1 + n4;
    if (need > stage_bytes) {
        if (stage) cudaFree(stage);
        stage = nullptr; stage_bytes = 0;
        if (cudaMalloc(&stage, need) != cudaSuccess) { cudaGetLastError(); return HTS_ERR_ALLOC; }
        stage_bytes = need;
    }
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    float* d_r = reinterpret_cast<float*>(stage);
    float* d_v = reinterpret_cast<float*>(stage + tn4);
    float* d_a = reinterpret_cast<float*>(stage + 2 * tn4);
    float* d_q = reinterpret_cast<float*>(stage + 3 * tn4);
    uint8_t* d_d = reinterpret_cast<uint8_t*>(stage + 4 * tn4);
    float* d_b = reinterpret_cast<float*>(stage + 4 * tn4 + tn1);
    HTS_CUDA(cudaMemcpyAsync(d_r, rewards, tn * 4, cudaMemcpyHostToDevice, s));
    HTS_CUDA(cudaMemcpyAsync(d_v, values, tn * 4, cudaMemcpyHostToDevice, s));
    HTS_CUDA(cudaMemcpyAsync(d_d, dones, tn, cudaMemcpyHostToDevice, s));
    HTS_CUDA(cudaMemcpyAsync(d_b, bootstrap, (size_t)N * 4, cudaMemcpyHostToDevice, s));
    st = launch_gae(d_r, d_v, d_d, d_b, gamma, lambda, T, N, d_a, d_q, s);
    if (st != HTS_OK) return st;
    HTS_CUDA(cudaMemcpyAsync(advantages, d_a, tn * 4, cudaMemcpyDeviceToHost, s));
    HTS_CUDA(cudaMemcpyAsync(returns, d_q, tn * 4, cudaMemcpyDeviceToHost, s));
    HTS_CUDA(cudaStreamSynchronize(s));
    return HTS_OK;
}

hts_status hts_gae_host_release(void)
{
    const int dev = device_slot();
    if (g_gae_stage[dev]) {
        HTS_CUDA(cudaDeviceSynchronize());
        HTS_CUDA(cudaFree(g_gae_stage[dev]));
        g_gae_stage[dev] = nullptr; g_gae_stage_bytes[dev] = 0;
    }
    return HTS_OK;
}

uint64_t hts_launch_count(void) { return hts::g_launches.load(std::memory_order_relaxed); }

const char* hts_last_cuda_error(void) { return hts::g_cuda_error; }

const char* hts_status_string(hts_status s)
{
    switch (s) {
        case HTS_OK: return "HTS_OK";
        case HTS_ERR_INVALID_ARG: return "HTS_ERR_INVALID_ARG";
        case HTS_ERR_SHAPE: return "HTS_ERR_SHAPE";
        case HTS_ERR_ALLOC: return "HTS_ERR_ALLOC";
        case HTS_ERR_CUDA: return "HTS_ERR_CUDA";
        case HTS_ERR_TIMEOUT: return "HTS_ERR_TIMEOUT";
        case HTS_ERR_UNSUPPORTED: return "HTS_ERR_UNSUPPORTED";
    }
    return "HTS_ERR_?";
}

}  // extern "C"
