// C ABI of the batch-1 decode step (see include/edgefm.h) and the launches of the step kernel.
#include "../../include/edgefm.h"

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "common.cuh"
#include "tensor_map.h"
#include "prefill.h"
#include "step_types.h"

namespace edgefm {

// ---- small kernels -------------------------------------------------------------------------------

// Strided copy of n caller-provided KV positions into cache slots [slot0, slot0 + n); also sets the device state
// (cache length slot0 + n).
__global__ void __launch_bounds__(256) prefill_copy_kernel(const uint16_t *k, const uint16_t *v, uint16_t *kc, uint16_t *vc,
                                                           int L, int nkv, int n, int d, int max_context, long long s_layer,
                                                           long long s_head, long long s_pos, int vec_ok, StepState *st, int slot0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->cur_len = slot0 + n;
        st->next_position = slot0 + n;
        if (st->status != STATUS_TIMEOUT) st->status = 0;
    }
    const long long total = static_cast<long long>(L) * nkv * n * d;
    const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
    if (vec_ok) {  // 16-byte pieces: d % 8 == 0, all strides % 8 == 0, bases 16-byte aligned
        const int dp = d >> 3;
        for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total >> 3; i += stride) {
            const int j = static_cast<int>(i % dp);
            long long r = i / dp;
            const int t = static_cast<int>(r % n); r /= n;
            const int g = static_cast<int>(r % nkv);
            const int l = static_cast<int>(r / nkv);
            const long long src = l * s_layer + g * s_head + t * s_pos + j * 8;
            const long long dst = ((static_cast<long long>(l) * nkv + g) * max_context + slot0 + t) * d + j * 8;
            *reinterpret_cast<uint4 *>(kc + dst) = *reinterpret_cast<const uint4 *>(k + src);
            *reinterpret_cast<uint4 *>(vc + dst) = *reinterpret_cast<const uint4 *>(v + src);
        }
    } else {
        for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < total; i += stride) {
            const int j = static_cast<int>(i % d);
            long long r = i / d;
            const int t = static_cast<int>(r % n); r /= n;
            const int g = static_cast<int>(r % nkv);
            const int l = static_cast<int>(r / nkv);
            const long long src = l * s_layer + g * s_head + t * s_pos + j;
            const long long dst = ((static_cast<long long>(l) * nkv + g) * max_context + slot0 + t) * d + j;
            kc[dst] = k[src];
            vc[dst] = v[src];
        }
    }
}

// The same for the compressed cache (Sec. 3.9): one warp per given row; the row's largest magnitude fixes its scale,
// scale = amax / 127, code = clamp(rint(x * (127 / amax))) in fp32.
__global__ void __launch_bounds__(256) prefill_quantize_kernel(const uint16_t *k, const uint16_t *v, signed char *kc, signed char *vc,
                                                               float *ks, float *vs, int L, int nkv, int n, int d, int max_context,
                                                               long long s_layer, long long s_head, long long s_pos, StepState *st,
                                                               int slot0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->cur_len = slot0 + n;
        st->next_position = slot0 + n;
        if (st->status != STATUS_TIMEOUT) st->status = 0;
    }
    const int warps = (gridDim.x * blockDim.x) >> 5, lane = threadIdx.x & 31;
    const long long rows = static_cast<long long>(L) * nkv * n * 2;          // K rows, then V rows
    for (long long r = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5; r < rows; r += warps) {
        const bool is_v = r >= rows / 2;
        long long rr = is_v ? r - rows / 2 : r;
        const int t = static_cast<int>(rr % n); rr /= n;
        const int g = static_cast<int>(rr % nkv);
        const int l = static_cast<int>(rr / nkv);
        const uint16_t *src = (is_v ? v : k) + l * s_layer + g * s_head + t * s_pos;
        const long long row = (static_cast<long long>(l) * nkv + g) * max_context + slot0 + t;
        float x[4];                                                          // d <= 128: at most 4 values per lane
        float amax = 0.f;
        for (int e = 0; e < 4; ++e) {
            const int j = lane + 32 * e;
            x[e] = j < d ? bf16_bits_to_f32(src[j]) : 0.f;
            amax = fmaxf(amax, fabsf(x[e]));
        }
        amax = warp_max(amax);
        const float inv = amax > 0.f ? __fdiv_rn(127.0f, amax) : 0.f;
        signed char *dst = (is_v ? vc : kc) + row * d;
        for (int e = 0; e < 4; ++e) {
            const int j = lane + 32 * e;
            if (j < d) dst[j] = static_cast<signed char>(static_cast<int>(fminf(fmaxf(rintf(__fmul_rn(x[e], inv)), -127.f), 127.f)));
        }
        if (lane == 0) (is_v ? vs : ks)[row] = amax > 0.f ? __fdiv_rn(amax, 127.0f) : 0.f;
    }
}

// Vocabulary pruning: row r of the compact lm_head is row ids[r] of the full one.  One warp per row, 16-byte pieces.
__global__ void __launch_bounds__(256) gather_rows_kernel(const uint16_t *src, const int *ids, uint16_t *dst, int n, int H) {
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int k16 = H >> 3;
    for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += warps) {
        const uint4 *s4 = reinterpret_cast<const uint4 *>(src + static_cast<size_t>(ids[r]) * H);
        uint4 *d4 = reinterpret_cast<uint4 *>(dst + static_cast<size_t>(r) * H);
        for (int c = lane; c < k16; c += 32) d4[c] = s4[c];
    }
}

// Raise the kernel's dynamic shared-memory limit to the most any plan can ask for (a function attribute, not an
// allocation).  Always the same value, so contexts and static calls of different shapes never lower it for one another.
inline cudaError_t allow_max_dynamic_smem(StepKernel kern, int smem_optin) {
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin - static_cast<int>(fa.sharedSizeBytes));
}

}  // namespace edgefm

using namespace edgefm;

// ---- the context -----------------------------------------------------------------------------------

struct edgefm_ctx {
    edgefm_shape shape{};
    int max_context = 0;
    int device = -1;
    int num_sms = 0;
    std::vector<edgefm_layer_weights> layers;
    const void *embed = nullptr, *final_norm = nullptr, *lm_head = nullptr;

    // owned device memory
    uint16_t *k_cache = nullptr, *v_cache = nullptr;  // [L][nkv][max_context][d] (bf16, or one signed byte per element)
    int kv_format = EDGEFM_KV_BF16;
    int block_tokens = 1;        // tokens a call may carry (edgefm_verify_block)
    float *k_scale = nullptr, *v_scale = nullptr;     // compressed cache: [L][nkv][max_context]
    double *inv_freq = nullptr;  // [d/2]
    StepState *state = nullptr;
    unsigned long long *prof = nullptr;
    int prof_stride = 0;

    // the persistent step kernel: the build for block_tokens tokens per call, and, from the first longer block on, the one for eight
    struct Build {
        StepLaunch launch;
        unsigned long long *ll = nullptr;     // exchange buffers
        unsigned char *maps = nullptr;        // tensor maps of the operators cut into boxes
        bool made = false;
    } step, wide;
    bool wide_refused = false;
    StepLayer *d_layers = nullptr;        // [n_layers + 1]
    // vocabulary pruning: the gathered rows of the current subset and their token ids
    int *vocab_ids = nullptr;       // [vocab]
    uint16_t *sub_lm = nullptr;     // [vocab_subset][hidden] or null
    int vocab_subset = 0;           // 0 = full vocabulary

    StepState *host_state = nullptr;      // pinned: edgefm_sync_length reads the device's state with one wait
    int launches_per_step = 0;
    PrefillBuffers pf;           // work buffers of edgefm_prefill, allocated at its first call
    int prefill_launches = 0;    // kernels the last edgefm_prefill (or block through the prompt kernels) enqueued
    uint32_t pf_wait_limit = 1u << 24, pf_extra_arrivals = 0;   // edgefm_debug_set_prefill_wait

    uint32_t spin_limit = 1000000000u;   // edgefm_debug_set_wait_limit: 1 s
    int barrier_extra = 0;

    // host mirrors
    int cur_len = 0;
    bool have_token = false;
    bool len_exact = true;       // false between a verified block (the device decides how far the cache grows) and edgefm_sync_length
    std::string err;
};

namespace {

thread_local std::string g_create_error;

edgefm_status fail(edgefm_ctx *ctx, edgefm_status st, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (ctx) ctx->err = buf; else g_create_error = buf;
    return st;
}

#define CUDA_TRY(ctx, call)                                                                                   \
    do {                                                                                                      \
        cudaError_t e_ = (call);                                                                              \
        if (e_ != cudaSuccess) {                                                                              \
            cudaGetLastError();   /* reported here: the check behind a later launch must not find it again */ \
            return fail(ctx, e_ == cudaErrorMemoryAllocation ? EDGEFM_ERR_OUT_OF_MEMORY : EDGEFM_ERR_CUDA,    \
                        "%s failed: %s", #call, cudaGetErrorString(e_));                                      \
        }                                                                                                     \
    } while (0)

struct DeviceGuard {
    int prev = -1;
    bool active = false;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) { cudaSetDevice(dev); active = true; }
    }
    ~DeviceGuard() { if (active) cudaSetDevice(prev); }
};

template <typename T>
cudaError_t dev_alloc(T **p, size_t count) {
    return cudaMalloc(reinterpret_cast<void **>(p), count * sizeof(T) + 256);  // + guard bytes behind every buffer
}

void free_all(edgefm_ctx *c) {
    for (edgefm_ctx::Build *b : {&c->step, &c->wide}) {
        if (b->ll) cudaFree(b->ll);
        if (b->maps) cudaFree(b->maps);
    }
    if (c->host_state) cudaFreeHost(c->host_state);
    void *bufs[] = {c->k_cache, c->v_cache, c->inv_freq, c->state, c->prof, c->vocab_ids, c->sub_lm, c->k_scale, c->v_scale, c->d_layers};
    for (void *b : bufs) if (b) cudaFree(b);
    if (c->pf.chunk) prefill_free(&c->pf);
}

edgefm_status ensure_prefill_buffers(edgefm_ctx *ctx);
PrefillModel prefill_model(edgefm_ctx *ctx);

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// One cooperative launch of the step kernel: all CTAs are co-resident, which the exchanges rely on.
cudaError_t launch_step(const StepLaunch &sl, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sl.grid);
    cfg.blockDim = dim3(ST_THREADS);
    cfg.dynamicSmemBytes = sl.dyn_smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, sl.kernel, sl.p);
}

// A step of a build: the request travels with the launch.
cudaError_t run_step(edgefm_ctx::Build *b, const StepRequest &r, cudaStream_t s) {
    b->launch.p.req = r;
    return launch_step(b->launch, s);
}

// Zeroed exchange buffers (with unit tables) and tensor maps of a build.  Enqueued on the stream of its first launch: the legacy stream is not
// ordered before a non-blocking one, nor the return of a pageable copy before its transfer.
cudaError_t init_build(const StepLaunch &sl, void *ll, void *maps, const void *host_maps, size_t map_bytes, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(ll, 0, sl.ll_bytes, s);
    // (pageable copies: the runtime stages the bytes before returning, so the sources may go)
    if (e == cudaSuccess) e = cudaMemcpyAsync(maps, host_maps, map_bytes, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess || !sl.unit_tab_bytes) return e;
    std::vector<unsigned> units(sl.unit_tab_bytes / 4);
    step_unit_table(sl, units.data());
    return cudaMemcpyAsync(const_cast<unsigned *>(sl.p.unit_tab), units.data(), sl.unit_tab_bytes, cudaMemcpyHostToDevice, s);
}

// Plan and buffers of the build for `mt` tokens per call, ready for launches on `s` (which is not being captured).  *why: the shape does not fit.
cudaError_t make_build(edgefm_ctx *c, int mt, edgefm_ctx::Build *b, cudaStream_t s, const char **why) {
    int smem_optin = 0, per_sm = 0;
    cudaError_t e = cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
    if (e != cudaSuccess) return e;
    StepLaunch &sl = b->launch;
    if ((*why = step_plan(c->shape, c->max_context, c->num_sms, smem_optin, c->kv_format == EDGEFM_KV_INT8, mt, &sl))) return cudaSuccess;
    if (!b->ll && (e = dev_alloc(&b->ll, sl.ll_bytes / 8)) != cudaSuccess) return e;
    step_wire(&sl, mt, b->ll);
    StepParams &p = sl.p;
    {
        std::vector<CUtensorMap> maps(static_cast<size_t>(4 * c->shape.n_layers) + 1);
        const bool sub = c->vocab_subset > 0;
        if (!step_maps(p, c->layers.data(), sub ? static_cast<const void *>(c->sub_lm) : c->lm_head, sub ? c->vocab_subset : c->shape.vocab, maps.data())) return cudaErrorUnknown;
        if (!b->maps && (e = cudaMalloc(reinterpret_cast<void **>(&b->maps), maps.size() * sizeof(CUtensorMap))) != cudaSuccess) return e;
        if ((e = init_build(sl, b->ll, b->maps, maps.data(), maps.size() * sizeof(CUtensorMap), s)) != cudaSuccess) return e;
        p.maps = b->maps;
        p.map_fence = 1;   // edgefm_set_vocab_subset rewrites the output layer's map
    }
    p.k_cache = c->k_cache; p.v_cache = c->v_cache; p.k_scale = c->k_scale; p.v_scale = c->v_scale;
    p.embed = static_cast<const uint16_t *>(c->embed); p.inv_freq = c->inv_freq; p.layers = c->d_layers; p.vocab_ids = c->vocab_ids;
    p.state = c->state; p.prof = c->prof; p.prof_stride = c->prof_stride;
    p.epoch_slot = b == &c->wide ? 1 : 0;
    p.spin_limit = c->spin_limit; p.barrier_extra = c->barrier_extra;
    if ((e = allow_max_dynamic_smem(sl.kernel, smem_optin)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sl.kernel, ST_THREADS, sl.dyn_smem)) != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidValue;
    c->launches_per_step = 1;
    b->made = true;
    return cudaSuccess;
}

}  // namespace

extern "C" {

const char *edgefm_version(void) { return "edgefm-b200 0.2 (sm_100a)"; }

const char *edgefm_last_error(const edgefm_ctx *ctx) { return ctx ? ctx->err.c_str() : g_create_error.c_str(); }

edgefm_status edgefm_create(const edgefm_shape *shape, const edgefm_weights *weights, int32_t max_context,
                            edgefm_ctx **out) {
    return edgefm_create_with_options(shape, weights, max_context, nullptr, out);
}

edgefm_status edgefm_create_with_options(const edgefm_shape *shape, const edgefm_weights *weights, int32_t max_context,
                                         const edgefm_options *options, edgefm_ctx **out) {
    if (out) *out = nullptr;
    if (options) {
        if (options->kv_format != EDGEFM_KV_BF16 && options->kv_format != EDGEFM_KV_INT8)
            return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "unknown kv_format %d", options->kv_format);
        for (int r : options->reserved)
            if (r != 0) return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "reserved option fields must be zero");
    }
    const bool kv8 = options && options->kv_format == EDGEFM_KV_INT8;
    if (options && options->block_tokens != 0 && options->block_tokens != 1 && options->block_tokens != 2 && options->block_tokens != 4)
        return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "block_tokens %d is not supported (0, 1, 2 or 4)", options->block_tokens);
    const int M = options && options->block_tokens > 1 ? options->block_tokens : 1;
    if (M > 1 && kv8) return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "blocks of several tokens need the plain bf16 cache");
    if (!shape || !weights || !out) return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "null argument");
    if (max_context < 1) return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "max_context must be >= 1");
    const edgefm_shape &sh = *shape;
    if (sh.n_layers < 1 || sh.hidden < 8 || sh.n_q_heads < 1 || sh.n_kv_heads < 1 || sh.ffn < 8 || sh.vocab < 1)
        return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "non-positive dimension");
    if (sh.hidden % 8 || sh.ffn % 8) return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "hidden and ffn must be multiples of 8");
    if (sh.head_dim != 64 && sh.head_dim != 128) return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "head_dim must be 64 or 128");
    if (sh.n_q_heads % sh.n_kv_heads) return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "n_q_heads must be a multiple of n_kv_heads");
    const int G = sh.n_q_heads / sh.n_kv_heads;
    if (G > 8) return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "group size n_q/n_kv must be <= 8");
    if (!(sh.rms_eps >= 0.f) || !(sh.rope_theta > 0.f)) return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "bad rms_eps / rope_theta");
    if (static_cast<long long>(sh.vocab) * sh.hidden > (1LL << 40)) return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "model too large");
    if (!weights->embed || !weights->final_norm || !weights->lm_head || !weights->layers)
        return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "null weight pointer");
    if (!aligned16(weights->embed) || !aligned16(weights->lm_head) || !aligned16(weights->final_norm))
        return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "weight pointers must be 16-byte aligned");
    for (int l = 0; l < sh.n_layers; ++l) {
        const edgefm_layer_weights &w = weights->layers[l];
        if (!w.input_norm || !w.wqkv || !w.wo || !w.post_norm || !w.w_gate_up || !w.w_down || (sh.qkv_bias && !w.bqkv))
            return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "null weight pointer in layer %d", l);
        if (!aligned16(w.input_norm) || !aligned16(w.wqkv) || !aligned16(w.wo) || !aligned16(w.post_norm) ||
            !aligned16(w.w_gate_up) || !aligned16(w.w_down))
            return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "weight pointers must be 16-byte aligned (layer %d)", l);
    }

    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return fail(nullptr, EDGEFM_ERR_CUDA, "no CUDA device available (this library has no CPU path)");
    }
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) {
        cudaGetLastError();
        return fail(nullptr, EDGEFM_ERR_CUDA, "cudaGetDeviceProperties failed");
    }
    if (prop.major < 10) return fail(nullptr, EDGEFM_ERR_CUDA, "device sm_%d%d is not supported (built for sm_100a)", prop.major, prop.minor);

    edgefm_ctx *c = new (std::nothrow) edgefm_ctx();
    if (!c) return fail(nullptr, EDGEFM_ERR_OUT_OF_MEMORY, "host allocation failed");
    c->shape = sh;
    c->kv_format = kv8 ? EDGEFM_KV_INT8 : EDGEFM_KV_BF16;
    c->block_tokens = M;
    c->max_context = max_context;
    c->device = dev;
    c->num_sms = prop.multiProcessorCount;
    c->layers.assign(weights->layers, weights->layers + sh.n_layers);
    c->embed = weights->embed; c->final_norm = weights->final_norm; c->lm_head = weights->lm_head;

    auto bail = [&](edgefm_status st, const char *what, cudaError_t e) {
        g_create_error = std::string(what) + ": " + cudaGetErrorString(e);
        cudaGetLastError();
        free_all(c);
        delete c;
        return st;
    };
#define CREATE_TRY(call)                                                                                            \
    do {                                                                                                            \
        cudaError_t e_ = (call);                                                                                    \
        if (e_ != cudaSuccess) return bail(e_ == cudaErrorMemoryAllocation ? EDGEFM_ERR_OUT_OF_MEMORY : EDGEFM_ERR_CUDA, #call, e_); \
    } while (0)

    const int d = sh.head_dim, nkv = sh.n_kv_heads;

    int coop = 0;
    CREATE_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    if (!coop) return bail(EDGEFM_ERR_CUDA, "device lacks cooperative launch", cudaErrorNotSupported);
    if (M > 1 && max_context > 8192) return bail(EDGEFM_ERR_BAD_SHAPE, "blocks of several tokens need max_context <= 8192", cudaErrorInvalidValue);

    const size_t kv_elems = static_cast<size_t>(sh.n_layers) * nkv * max_context * d;
    const size_t kv_bytes = kv8 ? kv_elems : kv_elems * 2;
    CREATE_TRY(dev_alloc(&c->k_cache, (kv_bytes + 1) / 2));
    CREATE_TRY(dev_alloc(&c->v_cache, (kv_bytes + 1) / 2));
    if (kv8) {
        const size_t kv_rows = static_cast<size_t>(sh.n_layers) * nkv * max_context;
        CREATE_TRY(dev_alloc(&c->k_scale, kv_rows));
        CREATE_TRY(dev_alloc(&c->v_scale, kv_rows));
        CREATE_TRY(cudaMemset(c->k_scale, 0, kv_rows * sizeof(float)));
        CREATE_TRY(cudaMemset(c->v_scale, 0, kv_rows * sizeof(float)));
    }
    CREATE_TRY(dev_alloc(&c->inv_freq, d / 2));
    CREATE_TRY(dev_alloc(&c->state, 1));
    CREATE_TRY(cudaHostAlloc(reinterpret_cast<void **>(&c->host_state), sizeof(StepState), cudaHostAllocDefault));
    CREATE_TRY(cudaMemset(c->k_cache, 0, kv_bytes));
    CREATE_TRY(cudaMemset(c->v_cache, 0, kv_bytes));
    CREATE_TRY(cudaMemset(c->state, 0, sizeof(StepState)));
    CREATE_TRY(dev_alloc(&c->vocab_ids, static_cast<size_t>(sh.vocab)));
    CREATE_TRY(cudaMemset(c->vocab_ids, 0, static_cast<size_t>(sh.vocab) * sizeof(int)));
    {
        std::vector<double> inv(d / 2);
        for (int i = 0; i < d / 2; ++i) inv[i] = std::pow(static_cast<double>(sh.rope_theta), -2.0 * i / d);
        CREATE_TRY(cudaMemcpy(c->inv_freq, inv.data(), inv.size() * sizeof(double), cudaMemcpyHostToDevice));
    }
    const char *pe_ = getenv("EDGEFM_PROFILE");
    if (pe_ && pe_[0] == '1') {
        c->prof_stride = 3 + 14 * sh.n_layers;
        const size_t n_prof = static_cast<size_t>(c->num_sms) * c->prof_stride;
        CREATE_TRY(dev_alloc(&c->prof, n_prof));
        CREATE_TRY(cudaMemset(c->prof, 0, n_prof * 8));
    }
    {
        std::vector<StepLayer> layers(static_cast<size_t>(sh.n_layers) + 1);
        step_layers(sh, c->layers.data(), c->final_norm, c->lm_head, layers.data());
        CREATE_TRY(dev_alloc(&c->d_layers, layers.size()));
        CREATE_TRY(cudaMemcpy(c->d_layers, layers.data(), layers.size() * sizeof(StepLayer), cudaMemcpyHostToDevice));
    }
    {
        const char *why = nullptr;
        CREATE_TRY(make_build(c, M, &c->step, nullptr, &why));
        if (why) return bail(EDGEFM_ERR_BAD_SHAPE, why, cudaErrorInvalidValue);
    }
    CREATE_TRY(cudaDeviceSynchronize());
#undef CREATE_TRY
    g_create_error.clear();
    *out = c;
    return EDGEFM_OK;
}

namespace {
// Common part of edgefm_prefill_kv (slot0 = 0) and edgefm_append_kv.
edgefm_status copy_kv_in(edgefm_ctx *ctx, const void *k, const void *v, int32_t slot0, int32_t n_positions, int64_t stride_layer,
                         int64_t stride_head, int64_t stride_pos, void *stream) {
    if (n_positions < 0) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "n_positions < 0");
    if (static_cast<int64_t>(slot0) + n_positions > ctx->max_context)
        return fail(ctx, EDGEFM_ERR_CONTEXT_FULL, "%d positions from slot %d exceed max_context %d", n_positions, slot0, ctx->max_context);
    if (n_positions > 0 && (!k || !v)) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "null k or v");
    if (n_positions > 0 && (stride_layer < 0 || stride_head < 0 || stride_pos < ctx->shape.head_dim))
        return fail(ctx, EDGEFM_ERR_INVALID_ARG, "bad strides");
    DeviceGuard guard(ctx->device);
    const edgefm_shape &sh = ctx->shape;
    if (ctx->kv_format == EDGEFM_KV_INT8) {
        long long blocks = (static_cast<long long>(sh.n_layers) * sh.n_kv_heads * n_positions * 2 + 7) / 8;   // 8 warps (rows) per block
        if (blocks < 1) blocks = 1;
        if (blocks > ctx->num_sms * 16) blocks = ctx->num_sms * 16;
        prefill_quantize_kernel<<<static_cast<unsigned>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const uint16_t *>(k), static_cast<const uint16_t *>(v), reinterpret_cast<signed char *>(ctx->k_cache),
            reinterpret_cast<signed char *>(ctx->v_cache), ctx->k_scale, ctx->v_scale, sh.n_layers, sh.n_kv_heads, n_positions, sh.head_dim,
            ctx->max_context, stride_layer, stride_head, stride_pos, ctx->state, slot0);
        CUDA_TRY(ctx, cudaGetLastError());
        ctx->cur_len = slot0 + n_positions;
        ctx->len_exact = true;
        ctx->err.clear();
        return EDGEFM_OK;
    }
    const int vec_ok = n_positions > 0 && aligned16(k) && aligned16(v) && stride_layer % 8 == 0 && stride_head % 8 == 0 &&
                       stride_pos % 8 == 0;
    const long long total = static_cast<long long>(sh.n_layers) * sh.n_kv_heads * n_positions * sh.head_dim;
    long long blocks = (total / (vec_ok ? 8 : 1) + 255) / 256;
    if (blocks < 1) blocks = 1;
    if (blocks > ctx->num_sms * 16) blocks = ctx->num_sms * 16;
    prefill_copy_kernel<<<static_cast<unsigned>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const uint16_t *>(k), static_cast<const uint16_t *>(v), ctx->k_cache, ctx->v_cache, sh.n_layers,
        sh.n_kv_heads, n_positions, sh.head_dim, ctx->max_context, stride_layer, stride_head, stride_pos, vec_ok, ctx->state, slot0);
    CUDA_TRY(ctx, cudaGetLastError());
    ctx->cur_len = slot0 + n_positions;
    ctx->len_exact = true;
    ctx->err.clear();
    return EDGEFM_OK;
}
}  // namespace

edgefm_status edgefm_prefill_kv(edgefm_ctx *ctx, const void *k, const void *v, int32_t n_positions, int64_t stride_layer,
                                int64_t stride_head, int64_t stride_pos, void *stream) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    return copy_kv_in(ctx, k, v, 0, n_positions, stride_layer, stride_head, stride_pos, stream);
}

edgefm_status edgefm_append_kv(edgefm_ctx *ctx, const void *k, const void *v, int32_t start, int32_t n_positions, int64_t stride_layer,
                               int64_t stride_head, int64_t stride_pos, void *stream) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (start < 0 || start > ctx->cur_len)
        return fail(ctx, EDGEFM_ERR_INVALID_ARG, "start %d outside [0, %d]: the cache may not have holes", start, ctx->cur_len);
    return copy_kv_in(ctx, k, v, start, n_positions, stride_layer, stride_head, stride_pos, stream);
}

edgefm_status edgefm_decode_step(edgefm_ctx *ctx, int32_t token_id, int32_t position, void *stream, float *logits_out,
                                 int32_t *next_token_out) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (token_id < -1 || token_id >= ctx->shape.vocab) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "token_id %d out of range", token_id);
    if (position < -1) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "position %d out of range", position);
    if (token_id == -1 && !ctx->have_token)
        return fail(ctx, EDGEFM_ERR_INVALID_ARG, "token_id -1 needs a previous step on this context");
    if (ctx->cur_len >= ctx->max_context)
        return fail(ctx, EDGEFM_ERR_CONTEXT_FULL, "KV cache is full (%d slots)", ctx->max_context);
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    StepRequest r{token_id, position, logits_out, next_token_out};
    CUDA_TRY(ctx, run_step(&ctx->step, r, s));
    ctx->cur_len += 1;
    ctx->have_token = true;
    ctx->err.clear();
    return EDGEFM_OK;
}

edgefm_status edgefm_verify_block(edgefm_ctx *ctx, const int32_t *tokens, int32_t m, int32_t position, void *stream, float *logits_out,
                                  int32_t *n_accepted_out, int32_t *next_token_out) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (!tokens) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "null tokens");
    const bool longer = m > ctx->block_tokens;   // than the context's build carries: the build for eight tokens, or the prompt kernels
    if (m < 1 || m > std::max(ctx->block_tokens, PF_VERIFY_MAX))
        return fail(ctx, EDGEFM_ERR_INVALID_ARG, "m = %d: blocks of 1 .. %d tokens", m, std::max(ctx->block_tokens, PF_VERIFY_MAX));
    if (longer && (tokens[0] < 0 || position < 0))
        return fail(ctx, EDGEFM_ERR_INVALID_ARG, "a block of %d tokens on this context (block_tokens = %d) needs tokens[0] and position given", m, ctx->block_tokens);
    if (longer && !ctx->len_exact)
        return fail(ctx, EDGEFM_ERR_INVALID_ARG, "the block is placed behind the host's cache length: call edgefm_sync_length after the previous block first");
    if (tokens[0] < -1 || tokens[0] >= ctx->shape.vocab) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "tokens[0] = %d out of range", tokens[0]);
    for (int t = 1; t < m; ++t)
        if (tokens[t] < 0 || tokens[t] >= ctx->shape.vocab) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "tokens[%d] = %d out of range", t, tokens[t]);
    if (position < -1) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "position %d out of range", position);
    if (tokens[0] == -1 && !ctx->have_token) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "tokens[0] = -1 needs a previous step on this context");
    if (ctx->cur_len + m > ctx->max_context)
        return fail(ctx, EDGEFM_ERR_CONTEXT_FULL, "%d tokens do not fit behind %d of %d cache slots", m, ctx->cur_len, ctx->max_context);
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    edgefm_ctx::Build *build = &ctx->step;
    bool prompt_kernels = longer && ctx->wide_refused;
    if (longer && !ctx->wide.made && !prompt_kernels) {
        // The build for eight tokens is made at the first longer block and kept, but not while a stream is being captured (it allocates)
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        CUDA_TRY(ctx, cudaStreamIsCapturing(s, &cap));
        if (cap != cudaStreamCaptureStatusNone) {
            prompt_kernels = true;
        } else {
            const char *why = nullptr;
            CUDA_TRY(ctx, make_build(ctx, PF_VERIFY_MAX, &ctx->wide, s, &why));
            prompt_kernels = ctx->wide_refused = why != nullptr;
        }
    }
    if (longer) build = &ctx->wide;
    if (prompt_kernels) {   // also for a shape whose vectors for eight tokens do not fit the shared memory
        if (const edgefm_status st = ensure_prefill_buffers(ctx)) return st;
        PrefillModel pm = prefill_model(ctx);
        int launches = 0;
        const int slot0 = ctx->cur_len;
        if (const char *e = prefill_run(pm, &ctx->pf, tokens, m, slot0, position, true, s, &launches)) {
            cudaGetLastError();
            return fail(ctx, EDGEFM_ERR_CUDA, "%s", e);
        }
        const bool sub = ctx->vocab_subset > 0;
        if (const char *e = prefill_verify_head(pm, &ctx->pf, m, ctx->final_norm, sub ? static_cast<const void *>(ctx->sub_lm) : ctx->lm_head,
                                                sub ? ctx->vocab_ids : nullptr, sub ? ctx->vocab_subset : ctx->shape.vocab, logits_out, n_accepted_out,
                                                next_token_out, slot0, position, s, &launches)) {
            cudaGetLastError();
            return fail(ctx, EDGEFM_ERR_CUDA, "%s", e);
        }
        ctx->prefill_launches = launches;
        ctx->cur_len += m;     // an upper bound until edgefm_sync_length
        ctx->len_exact = false;
        ctx->have_token = true;
        ctx->err.clear();
        return EDGEFM_OK;
    }
    StepRequest r{tokens[0], position, logits_out, next_token_out};
    r.m = m;
    for (int t = 1; t < m; ++t) r.draft[t - 1] = tokens[t];
    r.n_accepted_out = n_accepted_out;
    CUDA_TRY(ctx, run_step(build, r, s));
    ctx->cur_len += m;     // an upper bound until edgefm_sync_length: the device decides how many tokens are accepted
    if (m > 1) ctx->len_exact = false;
    ctx->have_token = true;
    ctx->err.clear();
    return EDGEFM_OK;
}

edgefm_status edgefm_prefill_tokens(edgefm_ctx *ctx, const int32_t *tokens, int32_t n, int32_t position, void *stream) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (n < 0 || (n > 0 && !tokens)) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "bad token list");
    if (position < 0) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "position %d out of range", position);
    for (int i = 0; i < n; ++i)
        if (tokens[i] < 0 || tokens[i] >= ctx->shape.vocab) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "tokens[%d] = %d out of range", i, tokens[i]);
    if (ctx->cur_len + n > ctx->max_context)
        return fail(ctx, EDGEFM_ERR_CONTEXT_FULL, "%d tokens do not fit behind %d of %d cache slots", n, ctx->cur_len, ctx->max_context);
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int M = ctx->block_tokens;
    for (int i = 0; i < n; i += M) {   // the step kernel, as many given tokens per call as the context's build carries
        const int m = n - i < M ? n - i : M;
        StepRequest r{tokens[i], position + i, nullptr, nullptr};
        r.m = m;
        for (int t = 1; t < m; ++t) r.draft[t - 1] = tokens[i + t];
        r.flags = 1;
        CUDA_TRY(ctx, run_step(&ctx->step, r, s));
        ctx->cur_len += m;
        ctx->have_token = true;
    }
    ctx->err.clear();
    return EDGEFM_OK;
}

}  // extern "C" (helpers of the prompt kernels follow)

namespace {

// Work buffers of the prompt kernels (prefill, verified blocks the step kernel does not take): allocated at the first use, kept.
edgefm_status ensure_prefill_buffers(edgefm_ctx *ctx) {
    if (ctx->pf.chunk == 0) {
        const int chunk = std::min(PF_CHUNK_MAX, ctx->max_context);
        if (prefill_alloc(&ctx->pf, ctx->shape, chunk, ctx->kv_format == EDGEFM_KV_INT8, ctx->num_sms) != cudaSuccess) {
            cudaGetLastError();
            prefill_free(&ctx->pf);
            return fail(ctx, EDGEFM_ERR_OUT_OF_MEMORY, "work buffers of the dense path (%zu bytes)", prefill_buffer_bytes(ctx->shape, chunk));
        }
    }
    ctx->pf.wait_limit = ctx->pf_wait_limit;
    ctx->pf.extra_arrivals = ctx->pf_extra_arrivals;
    return EDGEFM_OK;
}

PrefillModel prefill_model(edgefm_ctx *ctx) {
    return PrefillModel{ctx->shape, ctx->layers.data(), ctx->embed, ctx->k_cache, ctx->v_cache,
                        ctx->kv_format == EDGEFM_KV_INT8 ? ctx->k_scale : nullptr, ctx->kv_format == EDGEFM_KV_INT8 ? ctx->v_scale : nullptr,
                        ctx->max_context, ctx->state, ctx->num_sms};
}

}  // namespace

extern "C" {

edgefm_status edgefm_prefill(edgefm_ctx *ctx, const int32_t *tokens, int32_t n, int32_t position, void *stream, float *logits_out,
                             int32_t *next_token_out) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (n < 1 || !tokens) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "bad token list");
    if (position < 0) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "position %d out of range", position);
    for (int i = 0; i < n; ++i)
        if (tokens[i] < 0 || tokens[i] >= ctx->shape.vocab) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "tokens[%d] = %d out of range", i, tokens[i]);
    if (ctx->cur_len + n > ctx->max_context)
        return fail(ctx, EDGEFM_ERR_CONTEXT_FULL, "%d tokens do not fit behind %d of %d cache slots", n, ctx->cur_len, ctx->max_context);
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // Prompts of at least 8 tokens go through the dense path whole, and the output layer runs for the last row alone (one pass
    // over its matrix); shorter ones leave their last token to a decode step (which streams all weights again: 1.1 ms at the
    // 1.5B shape, against one more layer for a handful of rows).
    if (!ctx->len_exact)
        return fail(ctx, EDGEFM_ERR_INVALID_ARG, "the prompt is placed behind the host's cache length: call edgefm_sync_length after a verified block first");
    const bool dense_all = n >= 8;
    const int n_dense = dense_all ? n : n - 1;
    if (n_dense > 0)
        if (const edgefm_status st = ensure_prefill_buffers(ctx)) return st;
    PrefillModel pm = prefill_model(ctx);
    ctx->prefill_launches = 0;
    for (int i = 0; i < n_dense;) {
        const int c = std::min(ctx->pf.chunk, n_dense - i);
        int launches = 0;
        if (const char *e = prefill_run(pm, &ctx->pf, tokens + i, c, ctx->cur_len, position + i, dense_all && i + c == n_dense, s, &launches)) {
            cudaGetLastError();
            return fail(ctx, EDGEFM_ERR_CUDA, "%s", e);
        }
        ctx->prefill_launches += launches;
        ctx->cur_len += c;
        i += c;
        if (dense_all && i == n_dense) {   // the output layer for the prompt's last token, and the state a decode step would leave
            const bool sub = ctx->vocab_subset > 0;
            if (const char *e = prefill_head(pm, &ctx->pf, c - 1, ctx->final_norm, sub ? static_cast<const void *>(ctx->sub_lm) : ctx->lm_head,
                                             sub ? ctx->vocab_ids : nullptr, sub ? ctx->vocab_subset : ctx->shape.vocab, logits_out, next_token_out,
                                             tokens[n - 1], position + n - 1, s)) {
                cudaGetLastError();
                return fail(ctx, EDGEFM_ERR_CUDA, "%s", e);
            }
            ctx->prefill_launches += 1;
            ctx->have_token = true;
            ctx->err.clear();
            return EDGEFM_OK;
        }
    }
    const edgefm_status st = edgefm_decode_step(ctx, tokens[n - 1], position + n - 1, stream, logits_out, next_token_out);
    if (st == EDGEFM_OK) ctx->prefill_launches += ctx->launches_per_step;
    return st;
}

edgefm_status edgefm_sync_length(edgefm_ctx *ctx, void *stream, int32_t *cur_len_host) {
    if (!ctx || !cur_len_host) return EDGEFM_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    CUDA_TRY(ctx, cudaMemcpyAsync(ctx->host_state, ctx->state, sizeof(StepState), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(ctx, cudaStreamSynchronize(s));
    ctx->cur_len = ctx->host_state->cur_len;
    ctx->len_exact = true;
    *cur_len_host = ctx->cur_len;
    return EDGEFM_OK;
}

edgefm_status edgefm_destroy(edgefm_ctx *ctx) {
    if (!ctx) return EDGEFM_OK;
    DeviceGuard guard(ctx->device);
    cudaError_t e = cudaDeviceSynchronize();
    free_all(ctx);
    delete ctx;
    return e == cudaSuccess ? EDGEFM_OK : EDGEFM_ERR_CUDA;
}

edgefm_status edgefm_get_length(const edgefm_ctx *ctx, int32_t *cur_len_host) {
    if (!ctx || !cur_len_host) return EDGEFM_ERR_INVALID_ARG;
    *cur_len_host = ctx->cur_len;
    return EDGEFM_OK;
}

edgefm_status edgefm_set_vocab_subset(edgefm_ctx *ctx, const int32_t *token_ids, int32_t n, void *stream) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (n < 0 || n > ctx->shape.vocab) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "subset size %d outside [0, %d]", n, ctx->shape.vocab);
    if (n > 0 && !token_ids) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "null token_ids");
    for (int i = 0; i < n; ++i) {
        if (token_ids[i] < 0 || token_ids[i] >= ctx->shape.vocab)
            return fail(ctx, EDGEFM_ERR_INVALID_ARG, "token_ids[%d] = %d out of range", i, token_ids[i]);
        if (i > 0 && token_ids[i] <= token_ids[i - 1])
            return fail(ctx, EDGEFM_ERR_INVALID_ARG, "token_ids must be strictly ascending (entry %d)", i);
    }
    DeviceGuard guard(ctx->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int H = ctx->shape.hidden;
    uint16_t *fresh = nullptr;
    if (n > 0) CUDA_TRY(ctx, cudaMalloc(&fresh, static_cast<size_t>(n) * H * sizeof(uint16_t)));
    // steps already enqueued on the stream still read the previous subset
    cudaError_t e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && n > 0) {
        e = cudaMemcpyAsync(ctx->vocab_ids, token_ids, static_cast<size_t>(n) * sizeof(int32_t), cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) {
            int blocks = (n + 7) / 8;
            if (blocks > ctx->num_sms * 8) blocks = ctx->num_sms * 8;
            gather_rows_kernel<<<blocks, 256, 0, s>>>(static_cast<const uint16_t *>(ctx->lm_head), ctx->vocab_ids, fresh, n, H);
            e = cudaGetLastError();
        }
    }
    const uint16_t *lm_w = n > 0 ? fresh : static_cast<const uint16_t *>(ctx->lm_head);
    const StepHead head{lm_w, static_cast<const uint16_t *>(ctx->final_norm), n > 0 ? n : ctx->shape.vocab, n > 0 ? 1 : 0, {}};
    if (e == cudaSuccess) e = cudaMemcpyAsync(ctx->d_layers + ctx->shape.n_layers, &head, sizeof head, cudaMemcpyHostToDevice, s);
    CUtensorMap map[2];
    int k = 0;
    for (edgefm_ctx::Build *b : {&ctx->step, &ctx->wide}) {
        if (!b->made) continue;
        if (!step_map(&map[k], b->launch.p.cols[ST_LM], lm_w, head.rows)) e = cudaErrorUnknown;
        if (e == cudaSuccess) e = cudaMemcpyAsync(b->maps + static_cast<size_t>(4 * ctx->shape.n_layers) * sizeof(CUtensorMap), &map[k], sizeof(CUtensorMap), cudaMemcpyHostToDevice, s);
        ++k;
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // the host buffers are read before the call returns
    if (e != cudaSuccess) {
        if (fresh) cudaFree(fresh);
        return fail(ctx, EDGEFM_ERR_CUDA, "set_vocab_subset: %s", cudaGetErrorString(e));
    }
    if (ctx->sub_lm) cudaFree(ctx->sub_lm);
    ctx->sub_lm = fresh;
    ctx->vocab_subset = n;
    ctx->err.clear();
    return EDGEFM_OK;
}

edgefm_status edgefm_get_launches_per_step(const edgefm_ctx *ctx, int32_t *n) {
    if (!ctx || !n) return EDGEFM_ERR_INVALID_ARG;
    *n = ctx->launches_per_step;
    return EDGEFM_OK;
}

edgefm_status edgefm_get_prefill_launches(const edgefm_ctx *ctx, int32_t *n) {
    if (!ctx || !n) return EDGEFM_ERR_INVALID_ARG;
    *n = ctx->prefill_launches;
    return EDGEFM_OK;
}

edgefm_status edgefm_debug_profile(edgefm_ctx *ctx, uint64_t *out_host, int64_t capacity, int32_t *n_ctas, int32_t *stride) {
    if (!ctx || !n_ctas || !stride) return EDGEFM_ERR_INVALID_ARG;
    const int grid = ctx->step.launch.grid;
    *n_ctas = ctx->prof ? grid : 0;
    *stride = ctx->prof_stride;
    if (!ctx->prof || !out_host) return EDGEFM_OK;
    const int64_t n = static_cast<int64_t>(grid) * ctx->prof_stride;
    if (capacity < n) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "profile buffer too small");
    DeviceGuard guard(ctx->device);
    CUDA_TRY(ctx, cudaDeviceSynchronize());
    CUDA_TRY(ctx, cudaMemcpy(out_host, ctx->prof, static_cast<size_t>(n) * 8, cudaMemcpyDeviceToHost));
    return EDGEFM_OK;
}

edgefm_status edgefm_debug_plan(const edgefm_ctx *ctx, int32_t *out8) {
    if (!ctx || !out8) return EDGEFM_ERR_INVALID_ARG;
    const StepLaunch &sl = ctx->step.launch;
    const int32_t v[8] = {sl.grid, ST_NW, ST_BARS, sl.max_chunk_bytes, static_cast<int32_t>(sl.dyn_smem), sl.p.ring_bytes, sl.p.table_bytes, 0};
    std::copy(v, v + 8, out8);
    return EDGEFM_OK;
}

edgefm_status edgefm_debug_set_wait_limit(edgefm_ctx *ctx, uint32_t limit_ns, int32_t extra_barrier_arrivals) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (limit_ns < 1000u || extra_barrier_arrivals < 0 || extra_barrier_arrivals > 1)
        return fail(ctx, EDGEFM_ERR_INVALID_ARG, "limit_ns must be >= 1000 and extra_barrier_arrivals 0 or 1");
    DeviceGuard guard(ctx->device);
    CUDA_TRY(ctx, cudaDeviceSynchronize());
    ctx->spin_limit = limit_ns;
    ctx->barrier_extra = extra_barrier_arrivals;
    for (edgefm_ctx::Build *b : {&ctx->step, &ctx->wide}) {
        if (!b->made) continue;
        b->launch.p.spin_limit = limit_ns;
        b->launch.p.barrier_extra = extra_barrier_arrivals;
    }
    ctx->err.clear();
    return EDGEFM_OK;
}

edgefm_status edgefm_debug_set_prefill_wait(edgefm_ctx *ctx, uint32_t polls, int32_t extra_arrivals) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (polls < 1024u || extra_arrivals < 0 || extra_arrivals > 1)
        return fail(ctx, EDGEFM_ERR_INVALID_ARG, "polls must be >= 1024 and extra_arrivals 0 or 1");
    ctx->pf_wait_limit = polls;
    ctx->pf_extra_arrivals = static_cast<uint32_t>(extra_arrivals);
    ctx->err.clear();
    return EDGEFM_OK;
}

edgefm_status edgefm_debug_prefill_plan(int32_t epilogue, int32_t M, int32_t N, int32_t K, int32_t num_sms, int32_t *out2) {
    if (!out2 || epilogue < 0 || epilogue > 3 || M < 1 || N < 1 || K < 1 || num_sms < 1) return EDGEFM_ERR_INVALID_ARG;
    const PrefillPlan p = prefill_plan(epilogue == 3 ? 0 : epilogue, epilogue == 3 ? 64 : 128, M, N, K, num_sms);
    out2[0] = p.columns == 64 ? 2 : p.columns == 128 ? 0 : 1;
    out2[1] = p.cluster ? p.cluster : p.splits;
    return EDGEFM_OK;
}

edgefm_status edgefm_debug_prefill_launch(int32_t epilogue, int32_t M, int32_t N, int32_t K, int32_t num_sms, int32_t *out5) {
    if (!out5 || epilogue < 0 || epilogue > 3 || M < 1 || N < 1 || K < 1 || num_sms < 1) return EDGEFM_ERR_INVALID_ARG;
    const PrefillPlan p = prefill_plan(epilogue == 3 ? 0 : epilogue, epilogue == 3 ? 64 : 128, M, N, K, num_sms);
    out5[0] = p.columns;
    out5[1] = p.splits;
    out5[2] = p.cluster;
    out5[3] = p.pairs;
    out5[4] = p.swap;
    return EDGEFM_OK;
}

edgefm_status edgefm_debug_prefill_attention(int32_t T, int32_t slot0, int32_t n_q_heads, int32_t num_sms, int32_t *parts) {
    if (!parts || T < 1 || slot0 < 0 || n_q_heads < 1 || num_sms < 1) return EDGEFM_ERR_INVALID_ARG;
    *parts = prefill_attention_parts(T, slot0, n_q_heads, num_sms);
    return EDGEFM_OK;
}

edgefm_status edgefm_export_kv(edgefm_ctx *ctx, void *k_out, void *v_out, void *stream) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (!k_out || !v_out) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "null output");
    if (ctx->kv_format != EDGEFM_KV_BF16) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "this context has a compressed cache: use edgefm_export_kv_int8");
    DeviceGuard guard(ctx->device);
    const edgefm_shape &sh = ctx->shape;
    const size_t bytes = static_cast<size_t>(sh.n_layers) * sh.n_kv_heads * ctx->max_context * sh.head_dim * 2;
    CUDA_TRY(ctx, cudaMemcpyAsync(k_out, ctx->k_cache, bytes, cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream)));
    CUDA_TRY(ctx, cudaMemcpyAsync(v_out, ctx->v_cache, bytes, cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream)));
    return EDGEFM_OK;
}

edgefm_status edgefm_export_kv_int8(edgefm_ctx *ctx, void *k_codes_out, void *v_codes_out, float *k_scales_out, float *v_scales_out,
                                    void *stream) {
    if (!ctx) return EDGEFM_ERR_INVALID_ARG;
    if (!k_codes_out || !v_codes_out || !k_scales_out || !v_scales_out) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "null output");
    if (ctx->kv_format != EDGEFM_KV_INT8) return fail(ctx, EDGEFM_ERR_INVALID_ARG, "this context has the plain bf16 cache: use edgefm_export_kv");
    DeviceGuard guard(ctx->device);
    const edgefm_shape &sh = ctx->shape;
    const size_t rows = static_cast<size_t>(sh.n_layers) * sh.n_kv_heads * ctx->max_context;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CUDA_TRY(ctx, cudaMemcpyAsync(k_codes_out, ctx->k_cache, rows * sh.head_dim, cudaMemcpyDeviceToDevice, s));
    CUDA_TRY(ctx, cudaMemcpyAsync(v_codes_out, ctx->v_cache, rows * sh.head_dim, cudaMemcpyDeviceToDevice, s));
    CUDA_TRY(ctx, cudaMemcpyAsync(k_scales_out, ctx->k_scale, rows * sizeof(float), cudaMemcpyDeviceToDevice, s));
    CUDA_TRY(ctx, cudaMemcpyAsync(v_scales_out, ctx->v_scale, rows * sizeof(float), cudaMemcpyDeviceToDevice, s));
    return EDGEFM_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------------------
// edgefm_decode_step_static -- one decode step that allocates nothing.
//
// Some callers must not allocate device memory at all: a step issued from inside another framework's
// allocation-free region (a phase in which that framework has frozen its memory plan), from a process whose
// device memory is handed out entirely by a pool it does not own, or from a latency-critical thread where the
// implicit device synchronisation of cudaMalloc / cudaFree is not acceptable.  For them the work buffers of the
// persistent step kernel (residual stream, queries, attention partials, MLP activations, operator table, tile
// schedule, tensor maps, counters, device state: everything edgefm_create would allocate except the KV cache)
// live in a fixed array that is part of the loaded library image.  The caller owns the KV cache and the cache
// length and passes them in, so the call keeps no context.
//
// The array is EDGEFM_STATIC_SCRATCH_BYTES (4 MiB) on every GPU that loads the library, until exit.
namespace {

constexpr size_t EDGEFM_STATIC_SCRATCH_BYTES = 4u << 20;
static __device__ __align__(256) unsigned char g_static_scratch[EDGEFM_STATIC_SCRATCH_BYTES];

// In host code `g_static_scratch` is only a host-side stand-in for the symbol, not a device address.
// The device address is looked up once per device, with that device current.
constexpr int kMaxDevices = 64;
unsigned char *g_scratch_dev_ptr[kMaxDevices] = {};
StepState *g_static_state[kMaxDevices] = {};   // where the last static call on the device put its state word

struct ScratchCarver {
    unsigned char *base;
    size_t off = 0;
    template <typename T>
    T *take(size_t count) {
        T *p = reinterpret_cast<T *>(base + off);
        off = (off + count * sizeof(T) + 255) / 256 * 256;
        return p;
    }
};

}  // namespace

extern "C" edgefm_status edgefm_decode_step_static(const edgefm_shape *shape, const edgefm_weights *weights, void *k_cache,
                                                   void *v_cache, int32_t max_context, int32_t cur_len, int32_t token_id,
                                                   int32_t position, void *stream, float *logits_out,
                                                   int32_t *next_token_out) {
    if (!shape || !weights || !weights->layers || !k_cache || !v_cache)
        return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "null argument");
    const edgefm_shape &sh = *shape;
    constexpr int kMaxLayers = 96;
    if (sh.n_layers < 1 || sh.n_layers > kMaxLayers || sh.hidden < 8 || sh.hidden % 8 || sh.ffn < 8 || sh.ffn % 8 ||
        (sh.head_dim != 64 && sh.head_dim != 128) || sh.n_q_heads < 1 || sh.n_kv_heads < 1 || sh.n_q_heads % sh.n_kv_heads ||
        sh.n_q_heads / sh.n_kv_heads > 8 || sh.vocab < 1 || !(sh.rms_eps >= 0.f) || !(sh.rope_theta > 0.f))
        return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "unsupported model shape (same limits as edgefm_create; at most %d layers)", kMaxLayers);
    if (max_context < 1 || cur_len < 0 || cur_len >= max_context)
        return fail(nullptr, cur_len >= max_context ? EDGEFM_ERR_CONTEXT_FULL : EDGEFM_ERR_INVALID_ARG, "cur_len %d / max_context %d", cur_len, max_context);
    if (token_id < 0 || token_id >= sh.vocab || position < 0) return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "token or position out of range");
    if (!weights->embed || !weights->final_norm || !weights->lm_head) return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "null weight pointer");
    for (int l = 0; l < sh.n_layers; ++l) {
        const edgefm_layer_weights &w = weights->layers[l];
        if (!w.input_norm || !w.wqkv || !w.wo || !w.post_norm || !w.w_gate_up || !w.w_down || (sh.qkv_bias && !w.bqkv))
            return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "null weight pointer in layer %d", l);
        if (!aligned16(w.wqkv) || !aligned16(w.wo) || !aligned16(w.w_gate_up) || !aligned16(w.w_down) || !aligned16(w.input_norm) ||
            !aligned16(w.post_norm))
            return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "weight pointers must be 16-byte aligned (layer %d)", l);
    }
    if (!aligned16(weights->embed) || !aligned16(weights->lm_head) || !aligned16(weights->final_norm) || !aligned16(k_cache) || !aligned16(v_cache))
        return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "pointers must be 16-byte aligned");

    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return fail(nullptr, EDGEFM_ERR_CUDA, "no usable CUDA device (this library has no CPU path)");
    }
    // The small copies below read host buffers of this call; recorded into a capture they would be replayed from memory
    // that is gone by then.  A capturing stream is therefore refused before anything is enqueued.
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
            cudaGetLastError();
            return fail(nullptr, EDGEFM_ERR_CUDA, "cudaStreamIsCapturing failed");
        }
        if (cap != cudaStreamCaptureStatusNone)
            return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "edgefm_decode_step_static must not be called on a stream that is being captured");
    }
    const int d = sh.head_dim;
    int num_sms = 0, smem_optin = 0, coop = 0;
    CUDA_TRY(nullptr, cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev));
    CUDA_TRY(nullptr, cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    CUDA_TRY(nullptr, cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    if (!coop) return fail(nullptr, EDGEFM_ERR_CUDA, "device lacks cooperative launch");

    // ---- set-up, once per device: the device address of the scratch array (never the host-side symbol) ----
    if (!g_scratch_dev_ptr[dev]) {
        unsigned char *ptr = nullptr;
        CUDA_TRY(nullptr, cudaGetSymbolAddress(reinterpret_cast<void **>(&ptr), g_static_scratch));
        if (!ptr) return fail(nullptr, EDGEFM_ERR_CUDA, "cudaGetSymbolAddress returned a null scratch address");
        g_scratch_dev_ptr[dev] = ptr;
    }
    // ---- the same plan edgefm_create makes, in host memory -------------------------------------------------
    StepLaunch sl;
    if (const char *why = step_plan(sh, max_context, num_sms, smem_optin, false, 1, &sl)) return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "%s", why);

    // carve the scratch array; reject shapes that need more than it holds
    ScratchCarver sc{g_scratch_dev_ptr[dev]};
    StepLayer *d_layers = sc.take<StepLayer>(static_cast<size_t>(sh.n_layers) + 1);
    double *inv_freq = sc.take<double>(d / 2);
    StepState *state = sc.take<StepState>(1);
    CUtensorMap *d_maps = sc.take<CUtensorMap>(static_cast<size_t>(4 * sh.n_layers) + 1);
    unsigned long long *ll = sc.take<unsigned long long>(sl.ll_bytes / 8);
    if (sc.off > EDGEFM_STATIC_SCRATCH_BYTES)
        return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "this shape needs %zu bytes of work buffers; the static scratch holds %zu", sc.off,
                    EDGEFM_STATIC_SCRATCH_BYTES);
    std::vector<StepLayer> layers(static_cast<size_t>(sh.n_layers) + 1);
    step_layers(sh, weights->layers, weights->final_norm, weights->lm_head, layers.data());
    CUDA_TRY(nullptr, allow_max_dynamic_smem(sl.kernel, smem_optin));
    step_wire(&sl, 1, ll);
    StepParams &p = sl.p;
    p.k_cache = static_cast<uint16_t *>(k_cache); p.v_cache = static_cast<uint16_t *>(v_cache);
    p.embed = static_cast<const uint16_t *>(weights->embed); p.inv_freq = inv_freq; p.layers = d_layers;
    p.state = state;
    p.req = StepRequest{token_id, position, logits_out, next_token_out};
    p.maps = reinterpret_cast<const unsigned char *>(d_maps);
    p.map_fence = 2;   // every call rewrites all tensor maps in the shared scratch
    std::vector<CUtensorMap> maps(static_cast<size_t>(4 * sh.n_layers) + 1);
    if (!step_maps(p, weights->layers, weights->lm_head, sh.vocab, maps.data())) return fail(nullptr, EDGEFM_ERR_CUDA, "cuTensorMapEncodeTiled failed");

    // ---- stream-ordered set-up of the shared scratch: it still holds the previous call's contents ----------
    double inv[64];
    for (int i = 0; i < d / 2; ++i) inv[i] = std::pow(static_cast<double>(sh.rope_theta), -2.0 * i / d);
    StepState st{};
    st.cur_len = cur_len; st.next_position = position;
    // no packet of an earlier call (of any shape) may carry a tag of this one
    CUDA_TRY(nullptr, cudaMemsetAsync(ll, 0, sl.ll_bytes, s));
    std::vector<unsigned> units(sl.unit_tab_bytes / 4);
    if (!units.empty()) step_unit_table(sl, units.data());
    // pageable copies: the runtime stages the bytes before returning, so the sources may be freed after the call
    if (!units.empty()) CUDA_TRY(nullptr, cudaMemcpyAsync(const_cast<unsigned *>(p.unit_tab), units.data(), sl.unit_tab_bytes, cudaMemcpyHostToDevice, s));
    CUDA_TRY(nullptr, cudaMemcpyAsync(d_layers, layers.data(), layers.size() * sizeof(StepLayer), cudaMemcpyHostToDevice, s));
    CUDA_TRY(nullptr, cudaMemcpyAsync(d_maps, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice, s));
    CUDA_TRY(nullptr, cudaMemcpyAsync(inv_freq, inv, static_cast<size_t>(d / 2) * sizeof(double), cudaMemcpyHostToDevice, s));
    CUDA_TRY(nullptr, cudaMemcpyAsync(state, &st, sizeof st, cudaMemcpyHostToDevice, s));
    CUDA_TRY(nullptr, launch_step(sl, s));
    g_static_state[dev] = state;
    g_create_error.clear();
    return EDGEFM_OK;
}

extern "C" edgefm_status edgefm_sync_status(edgefm_ctx *ctx, void *stream) {
    // ctx == NULL: the status word the last edgefm_decode_step_static on the current device left in the static scratch
    int dev = -1;
    StepState *where = nullptr;
    if (ctx) {
        where = ctx->state;
    } else {
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices || !g_static_state[dev]) {
            cudaGetLastError();
            return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "no static step has run on the current device");
        }
        where = g_static_state[dev];
    }
    DeviceGuard guard(ctx ? ctx->device : dev);
    CUDA_TRY(ctx, cudaStreamSynchronize(static_cast<cudaStream_t>(stream)));
    StepState st;
    CUDA_TRY(ctx, cudaMemcpy(&st, where, sizeof st, cudaMemcpyDeviceToHost));
    if (ctx && ctx->pf.chunk) {
        int pe = 0;
        CUDA_TRY(ctx, cudaMemcpy(&pe, ctx->pf.error, sizeof pe, cudaMemcpyDeviceToHost));
        if (pe != 0) return fail(ctx, EDGEFM_ERR_TIMEOUT, "a bounded wait of a prefill contraction expired; the context must be destroyed");
    }
    if (st.status != 0)
        return fail(ctx, EDGEFM_ERR_TIMEOUT, "device status %d (6 = a bounded wait expired, 100+ = self-check code) operands %d %d; "
                    "the context must be destroyed", st.status, st.pad[0], st.pad[1]);
    return EDGEFM_OK;
}

// Host-only diagnostics: the plan of the step kernel for a shape, and the chunks one CTA streams of one operator, with the kernel's own arithmetic.
extern "C" edgefm_status edgefm_debug_step_plan(const edgefm_shape *shape, int32_t max_context, int32_t kv_format, int32_t tokens, int32_t n_sms, int32_t smem_bytes,
                                                int32_t *out40, int32_t op, int32_t cta, uint32_t *chunks_out, int32_t capacity, int32_t *n_chunks) {
    if (!shape || !out40 || !n_chunks || max_context < 1 || n_sms < 1 || op < 0 || op > ST_LM || cta < 0) return fail(nullptr, EDGEFM_ERR_INVALID_ARG, "bad argument");
    const edgefm_shape &sh = *shape;
    if (sh.n_layers < 1 || sh.hidden < 8 || sh.hidden % 8 || sh.ffn < 8 || sh.ffn % 8 || (sh.head_dim != 64 && sh.head_dim != 128) || sh.n_q_heads < 1 || sh.n_kv_heads < 1 ||
        sh.n_q_heads % sh.n_kv_heads || sh.n_q_heads / sh.n_kv_heads > 8 || sh.vocab < 1)
        return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "unsupported model shape");
    StepLaunch sl;
    if (const char *why = step_plan(sh, max_context, n_sms, smem_bytes, kv_format == EDGEFM_KV_INT8, tokens, &sl)) return fail(nullptr, EDGEFM_ERR_BAD_SHAPE, "%s", why);
    const StepParams &p = sl.p;
    const int32_t head[15] = {sl.grid, static_cast<int32_t>(sl.dyn_smem), p.ring_bytes, sl.max_chunk_bytes, p.table_bytes, sl.list_len, sl.list_len == 0, static_cast<int32_t>(sl.unit_tab_bytes),
                              p.kv_block, p.act_slots, p.act_packets, p.merged_len, p.act_len, p.x_line, p.ao_line};
    std::copy(head, head + 15, out40);
    for (int o = 0; o < 5; ++o) {
        const StepCols &c = p.cols[o];
        const int32_t v[5] = {c.K, c.seg, c.segs, c.box_rows, c.tile};
        std::copy(v, v + 5, out40 + 15 + 5 * o);
    }
    *n_chunks = cta < sl.grid ? step_chunks(sl, op, cta, chunks_out, chunks_out ? capacity : 0) : 0;
    return EDGEFM_OK;
}
