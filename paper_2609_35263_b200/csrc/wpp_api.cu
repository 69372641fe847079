// C-ABI entry points that touch CUDA: context, tensor-map construction, argument checks and launches.
// There is no CPU fallback: without a usable device wpp_create fails and nothing else can be called.
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>
#include <new>

#include "../../include/wpp.h"
#include "wpp_device.h"
#include "wpp_host.h"
#include "wpp_plan_format.h"

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// A tensor map depends only on (base pointer, extents, strides, box); serving loops call with the same pools and
// the same query buffers wave after wave, so the context keeps the maps it has encoded.
struct MapKey {
    const void* base;
    uint64_t dims[4], strides[3];
    uint32_t box[4];
    int rank, swizzle;
};
struct MapEntry {
    MapKey key;
    CUtensorMap map;
    uint64_t used;      // 0 = empty; else the tick of the last use (least recently used entry is replaced)
};
constexpr int kMapCacheEntries = 32;
constexpr int kLateRescaleOnPct = 30, kLateRescaleOffPct = 15;   // share of key steps that rescale O (see choose_late_rescale)

struct wpp_ctx {
    int device;
    int sm_count;
    int smem_optin;
    int last_cuda_error;
    int64_t launches;
    EncodeTiledFn encode_tiled;
    void* static_scratch;           // device address of the built-in scratch array on this context's device
    // Where a moved row reference rescales O (see the attention kernel's kLate) is chosen per launch from what the
    // kernels of earlier launches counted: key steps and steps that rescaled.
    int counters;                   // which of the device's counters are this context's, -1: none
    volatile unsigned long long* totals_host;    // [kCounterSlots][2]: totals that launches have left, as the host sees them
    char* totals_dev;               // the same as the device sees them
    uint32_t next_slot;             // launches in turn
    unsigned long long steps, moves;             // the largest totals seen so far ...
    unsigned long long base_steps, base_moves;   // ... and those at the context's creation
    unsigned long long seen_steps, seen_moves;   // the counters when the choice was last looked at
    int rescale_mode;               // 0: always before the exponentials (default), 1: always after, 2: chosen from the counters
    int late_rescale;               // the current choice
    std::mutex* map_lock;
    uint64_t map_tick;
    MapEntry maps[kMapCacheEntries];
};

// ---------------------------------------------------------------------------------------------------------------
// Built-in scratch for the entry point that allocates nothing (wpp_prefill_attention_varlen_static, below).
// Some callers of this library cannot call cudaMalloc when a wave is due: the serving process has handed all free
// device memory to the KV page pool, and an allocation on the execution path would fail or stall the stream.
#define WPP_STATIC_SCRATCH_BYTES (16u << 20)
static __device__ __align__(256) unsigned char wpp_static_scratch[WPP_STATIC_SCRATCH_BYTES];

extern "C" size_t wpp_static_scratch_bytes(void) { return (size_t)WPP_STATIC_SCRATCH_BYTES; }

// In host code the array's name is only a handle, not a device address.  The address is looked up once per
// device, with that device current (the symbol resolves to the current device's copy).  The look-up is also
// what makes the CUDA runtime load this module on the device, i.e. what reserves the 16 MiB there: it runs
// inside wpp_create, at start-up, so that no later call has to find memory for it.
static std::mutex g_scratch_lock;
static void* g_scratch_ptr[64];

static cudaError_t static_scratch_address(int device, void** out) {
    std::lock_guard<std::mutex> guard(g_scratch_lock);
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    if (!g_scratch_ptr[device]) {
        int cur = -1;
        cudaError_t e = cudaGetDevice(&cur);
        if (e != cudaSuccess) return e;
        if (cur != device && (e = cudaSetDevice(device)) != cudaSuccess) return e;
        void* ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, wpp_static_scratch);
        if (cur != device) cudaSetDevice(cur);
        if (e != cudaSuccess) return e;
        if (!ptr) return cudaErrorInvalidSymbol;
        g_scratch_ptr[device] = ptr;
    }
    *out = g_scratch_ptr[device];
    return cudaSuccess;
}

// The counters of the contexts on a device: device memory of the attention kernel's module, and pinned memory mapped for the
// device, to which the kernels store totals: allocated with the first context on a device, kept, and aligned to its size, so that
// an address in it says which context's counters and which slot it stands for.  Contexts beyond kCounterContexts at a time on
// a device have none (their choice of order stays at its default).
struct CounterPool {
    char *host, *dev;
    bool used[wpp::kCounterContexts];
};
static CounterPool g_counters[64];

// (no CUDA call but for the first context on a device)
static void take_counters(wpp_ctx* c) {
    c->counters = -1;
    std::lock_guard<std::mutex> guard(g_scratch_lock);
    if (c->device < 0 || c->device >= 64) return;
    CounterPool& pool = g_counters[c->device];
    if (!pool.host) {
        constexpr uintptr_t size = wpp::kCounterBytes;
        int before = -1;
        void *host = nullptr, *dev = nullptr;
        if (cudaGetDevice(&before) != cudaSuccess) return;
        if (before != c->device && cudaSetDevice(c->device) != cudaSuccess) return;
        if (cudaHostAlloc(&host, 2 * size, cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess) {
            char* at = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(host) + size - 1) / size * size);
            if (cudaHostGetDevicePointer(&dev, at, 0) == cudaSuccess && reinterpret_cast<uintptr_t>(dev) % size == 0) {
                memset(at, 0, size);
                pool.host = at;
                pool.dev = static_cast<char*>(dev);
            } else {
                cudaFreeHost(host);
            }
        }
        if (before != c->device) cudaSetDevice(before);
        (void)cudaGetLastError();
    }
    for (int i = 0; pool.host && i < wpp::kCounterContexts; ++i) {
        if (pool.used[i]) continue;
        pool.used[i] = true;
        c->counters = i;
        const size_t off = (size_t)i * wpp::kCounterSlots * 16;
        c->totals_host = reinterpret_cast<volatile unsigned long long*>(pool.host + off);
        c->totals_dev = pool.dev + off;
        return;
    }
}
static void give_counters_back(const wpp_ctx* c) {
    if (c->counters < 0) return;
    std::lock_guard<std::mutex> guard(g_scratch_lock);
    g_counters[c->device].used[c->counters] = false;
}

// The totals now: every launch leaves them at its end, in a slot of its own, so the largest are the newest (map_lock is held).
static void read_counters(wpp_ctx* c) {
    for (int i = 0; c->counters >= 0 && i < wpp::kCounterSlots; ++i) {
        const unsigned long long steps = c->totals_host[2 * i], moves = c->totals_host[2 * i + 1];
        if (steps > c->steps || (steps == c->steps && moves > c->moves)) {
            c->steps = steps;
            if (moves > c->moves) c->moves = moves;
        }
    }
}

// Creating a context must neither disturb a stream that is being captured nor be refused for it.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

extern "C" int wpp_ctx_sm_count(const wpp_ctx* ctx) { return ctx ? ctx->sm_count : 148; }

static int cuda_fail(const wpp_ctx* ctx, int err) {
    if (ctx) const_cast<wpp_ctx*>(ctx)->last_cuda_error = err;
    return WPP_ERR_CUDA;
}

extern "C" int wpp_create(wpp_ctx** out, int cuda_device) {
    if (!out) return WPP_ERR_INVALID_ARG;
    *out = nullptr;
    RelaxedCapture relaxed;
    int n = 0;
    cudaError_t e = cudaGetDeviceCount(&n);
    if (e != cudaSuccess || cuda_device < 0 || cuda_device >= n) return WPP_ERR_CUDA;
    cudaDeviceProp prop;
    if ((e = cudaGetDeviceProperties(&prop, cuda_device)) != cudaSuccess) return WPP_ERR_CUDA;
    if (prop.major != 10) return WPP_ERR_UNSUPPORTED;   // the kernels are built for sm_100a only
    wpp_ctx* c = static_cast<wpp_ctx*>(calloc(1, sizeof(wpp_ctx)));
    if (!c) return WPP_ERR_INVALID_ARG;
    c->device = cuda_device;
    c->sm_count = prop.multiProcessorCount;
    c->smem_optin = (int)prop.sharedMemPerBlockOptin;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
    if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || !fn) {
        free(c);
        return WPP_ERR_CUDA;
    }
    c->encode_tiled = reinterpret_cast<EncodeTiledFn>(fn);
    if (static_scratch_address(cuda_device, &c->static_scratch) != cudaSuccess) {
        free(c);
        return WPP_ERR_CUDA;
    }
    c->map_lock = new (std::nothrow) std::mutex();
    if (!c->map_lock) {
        free(c);
        return WPP_ERR_INVALID_ARG;
    }
    take_counters(c);
    read_counters(c);
    c->base_steps = c->seen_steps = c->steps;
    c->base_moves = c->seen_moves = c->moves;
    *out = c;
    return WPP_OK;
}

// (no CUDA call: a context may be collected while a stream is being captured)
extern "C" int wpp_destroy(wpp_ctx* ctx) {
    if (ctx) {
        give_counters_back(ctx);
        delete ctx->map_lock;
    }
    free(ctx);
    return WPP_OK;
}

extern "C" int wpp_set_rescale_mode(wpp_ctx* ctx, int mode) {
    if (!ctx || mode < 0 || mode > 2) return WPP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> guard(*ctx->map_lock);
    ctx->rescale_mode = mode;
    return WPP_OK;
}

extern "C" int wpp_rescale_stats(const wpp_ctx* ctx, uint64_t* key_steps, uint64_t* rescaling_steps, int* late) {
    if (!ctx) return WPP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> guard(*ctx->map_lock);
    read_counters(const_cast<wpp_ctx*>(ctx));
    if (key_steps) *key_steps = ctx->steps - ctx->base_steps;
    if (rescaling_steps) *rescaling_steps = ctx->moves - ctx->base_moves;
    if (late) *late = ctx->rescale_mode == 1 || (ctx->rescale_mode == 2 && ctx->late_rescale);
    return WPP_OK;
}

// The choice for the next launch, and in *totals where it leaves the totals: with the counters' increase since the last look,
// once there are enough steps to judge by; between the two thresholds the choice stays what it was.
static int choose_late_rescale(const wpp_ctx* cctx, unsigned long long** totals) {
    wpp_ctx* c = const_cast<wpp_ctx*>(cctx);
    std::lock_guard<std::mutex> guard(*c->map_lock);
    *totals = nullptr;
    if (c->counters >= 0) *totals = reinterpret_cast<unsigned long long*>(c->totals_dev + 16 * (c->next_slot++ % wpp::kCounterSlots));
    if (c->rescale_mode != 2) return c->rescale_mode == 1;
    read_counters(c);
    const unsigned long long ds = c->steps - c->seen_steps, dm = c->moves - c->seen_moves;
    if (ds >= 4096) {
        if (dm * 100 >= ds * kLateRescaleOnPct) c->late_rescale = 1;
        else if (dm * 100 < ds * kLateRescaleOffPct) c->late_rescale = 0;
        c->seen_steps = c->steps;
        c->seen_moves = c->moves;
    }
    return c->late_rescale;
}

// Every launching entry point runs with the context's device current: a call made with another device current
// would launch there with this device's pointers and tensor maps.
extern "C" int wpp_ctx_check_device(const wpp_ctx* ctx) {
    int cur = -1;
    cudaError_t e = cudaGetDevice(&cur);
    if (e != cudaSuccess) return cuda_fail(ctx, (int)e);
    return cur == ctx->device ? WPP_OK : WPP_ERR_INVALID_ARG;
}

extern "C" int wpp_last_cuda_error(const wpp_ctx* ctx) { return ctx ? ctx->last_cuda_error : 0; }
extern "C" int64_t wpp_launch_count(const wpp_ctx* ctx) { return ctx ? ctx->launches : 0; }

extern "C" int wpp_selftest_bounded_wait(const wpp_ctx* ctx, int64_t limit_cycles, int32_t* status_dev,
                                         int64_t* waited_cycles_dev, void* cuda_stream) {
    if (!ctx || !status_dev || limit_cycles < 1 || limit_cycles > (1ll << 30)) return WPP_ERR_INVALID_ARG;
    if (int rc = wpp_ctx_check_device(ctx)) return rc;
    int e = wpp_launch_selftest_wait((long long)limit_cycles, status_dev,
                                     reinterpret_cast<long long*>(waited_cycles_dev), cuda_stream);
    if (e != 0) return cuda_fail(ctx, e);
    const_cast<wpp_ctx*>(ctx)->launches += 1;
    return WPP_OK;
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// bf16 tensor map, with 128-byte swizzle unless told otherwise; dims/strides innermost first, strides in bytes for dims 1..rank-1.
// Looked up in the context's cache first (six maps per attention call; encoding them costs more than a small
// wave's kernel).
static int make_map(const wpp_ctx* cctx, CUtensorMap* m, const void* base, int rank, const uint64_t* dims,
                    const uint64_t* strides_bytes, const uint32_t* box, bool swizzle = true) {
    wpp_ctx* ctx = const_cast<wpp_ctx*>(cctx);
    MapKey key;
    memset(&key, 0, sizeof(key));
    key.base = base;
    key.rank = rank;
    key.swizzle = swizzle;
    for (int i = 0; i < rank; ++i) { key.dims[i] = dims[i]; key.box[i] = box[i]; }
    for (int i = 0; i < rank - 1; ++i) key.strides[i] = strides_bytes[i];
    std::lock_guard<std::mutex> guard(*ctx->map_lock);
    const uint64_t tick = ++ctx->map_tick;
    int victim = 0;
    for (int i = 0; i < kMapCacheEntries; ++i) {
        MapEntry& en = ctx->maps[i];
        if (en.used && memcmp(&en.key, &key, sizeof(key)) == 0) {
            en.used = tick;
            *m = en.map;
            return WPP_OK;
        }
        if (en.used < ctx->maps[victim].used) victim = i;
    }
    cuuint64_t gd[4];
    cuuint64_t gs[3];
    cuuint32_t bx[4], es[4];
    for (int i = 0; i < rank; ++i) { gd[i] = dims[i]; bx[i] = box[i]; es[i] = 1; }
    for (int i = 0; i < rank - 1; ++i) gs[i] = strides_bytes[i];
    CUresult r = ctx->encode_tiled(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), gd,
                                   gs, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cuda_fail(ctx, (int)r);
    MapEntry& en = ctx->maps[victim];
    memcpy(&en.key, &key, sizeof(key));
    en.map = *m;
    en.used = tick;
    return WPP_OK;
}

extern "C" int wpp_kv_append(const wpp_ctx* ctx, const wpp_batch_desc* desc, const void* k_new, const void* v_new,
                             void* k_cache, void* v_cache, const int32_t* block_tables, const int32_t* prefix_lens,
                             const int32_t* chunk_lens, const void* plan_host, const void* plan_dev,
                             int32_t* status_dev, void* cuda_stream) {
    if (!ctx) return WPP_ERR_INVALID_ARG;
    wpp_batch_desc d;
    int rc = wpp_resolve_desc(desc, &d);
    if (rc != WPP_OK) return rc;
    const WppPlanHeader* hd = nullptr;
    if ((rc = wpp_check_plan(plan_host, &d, &hd)) != WPP_OK) return rc;
    if (hd->total_new_tokens == 0) return WPP_OK;
    if ((rc = wpp_ctx_check_device(ctx)) != WPP_OK) return rc;
    if (!k_new || !v_new || !k_cache || !v_cache || !block_tables || !prefix_lens || !chunk_lens || !plan_dev)
        return WPP_ERR_INVALID_ARG;
    if (!aligned16(k_new) || !aligned16(v_new) || !aligned16(k_cache) || !aligned16(v_cache) || !aligned16(plan_dev))
        return WPP_ERR_INVALID_ARG;
    wpp::AppendParams p;
    memset(&p, 0, sizeof(p));
    p.plan = plan_dev;
    p.k_new = static_cast<const uint4*>(k_new);
    p.v_new = static_cast<const uint4*>(v_new);
    p.k_cache = static_cast<uint4*>(k_cache);
    p.v_cache = static_cast<uint4*>(v_cache);
    p.block_tables = block_tables;
    p.prefix_lens = prefix_lens;
    p.chunk_lens = chunk_lens;
    p.status = status_dev;
    p.kvnew_token_stride = d.kvnew_token_stride / 8;
    p.kvnew_head_stride = d.kvnew_head_stride / 8;
    p.kv_page_stride = d.kv_page_stride / 8;
    p.kv_head_stride = d.kv_head_stride / 8;
    p.kv_token_stride = d.kv_token_stride / 8;
    p.num_requests = d.num_requests;
    p.num_kv_heads = d.num_kv_heads;
    p.vec_per_row = d.head_dim / 8;
    p.page_size = d.page_size;
    p.max_blocks = d.max_blocks_per_req;
    p.num_pages = d.num_pages;
    p.total_new_tokens = hd->total_new_tokens;
    p.off_q_offsets = hd->off_q_offsets;
    p.off_prefix = hd->off_prefix;
    int e = wpp_launch_append(&p, ctx->sm_count, cuda_stream);
    if (e != 0) return cuda_fail(ctx, e);
    const_cast<wpp_ctx*>(ctx)->launches += 1;
    return WPP_OK;
}

extern "C" int wpp_prefill_attention_varlen(const wpp_ctx* ctx, const wpp_batch_desc* desc, const void* q, void* out,
                                            float* lse_or_null, const void* k_cache, const void* v_cache,
                                            const int32_t* block_tables, const int32_t* prefix_lens,
                                            const int32_t* chunk_lens, const void* plan_host, const void* plan_dev,
                                            void* workspace, size_t workspace_bytes, int32_t* status_dev,
                                            void* cuda_stream) {
    if (!ctx) return WPP_ERR_INVALID_ARG;
    wpp_batch_desc d;
    int rc = wpp_resolve_desc(desc, &d);
    if (rc != WPP_OK) return rc;
    const WppPlanHeader* hd = nullptr;
    if ((rc = wpp_check_plan(plan_host, &d, &hd)) != WPP_OK) return rc;
    if (hd->tile_m > WPP_MAX_TILE_M || hd->shape < 1 || hd->shape > 2) return WPP_ERR_PLAN_MISMATCH;
    if (hd->total_new_tokens == 0 || hd->num_units == 0) return WPP_OK;
    if ((rc = wpp_ctx_check_device(ctx)) != WPP_OK) return rc;
    if (!q || !out || !k_cache || !v_cache || !block_tables || !prefix_lens || !chunk_lens || !plan_dev)
        return WPP_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(out) || !aligned16(k_cache) || !aligned16(v_cache) || !aligned16(plan_dev))
        return WPP_ERR_INVALID_ARG;
    // the workspace always holds the tile counter, and the split partials behind it when the plan has any
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0) return WPP_ERR_INVALID_ARG;
    if (workspace_bytes < hd->workspace_bytes) return WPP_ERR_WORKSPACE_TOO_SMALL;
    if (d.num_pages == 0) return WPP_ERR_INVALID_ARG;

    CUtensorMap tq[4], tk, tv;
    for (int i = 0; i < 4; ++i) {       // boxes of 128, 64, 32, 16 query rows (packed heads take fewer rows per head)
        const uint64_t dims[3] = {(uint64_t)d.head_dim, (uint64_t)d.num_q_heads, (uint64_t)hd->total_new_tokens};
        const uint64_t strides[2] = {(uint64_t)d.q_head_stride * 2, (uint64_t)d.q_token_stride * 2};
        const uint32_t box[3] = {64, 1, (uint32_t)(128 >> i)};
        if ((rc = make_map(ctx, &tq[i], q, 3, dims, strides, box)) != WPP_OK) return rc;
    }
    {
        const uint64_t dims[4] = {(uint64_t)d.head_dim, (uint64_t)d.page_size, (uint64_t)d.num_kv_heads,
                                  (uint64_t)d.num_pages};
        const uint64_t strides[3] = {(uint64_t)d.kv_token_stride * 2, (uint64_t)d.kv_head_stride * 2,
                                     (uint64_t)d.kv_page_stride * 2};
        // the small shape works on 64-key steps: its boxes have at most 64 rows (half a 128-token page)
        const uint32_t box_rows = (hd->shape == 2 && d.page_size > 64) ? 64u : (uint32_t)d.page_size;
        const uint32_t box[4] = {64, box_rows, 1, 1};
        if ((rc = make_map(ctx, &tk, k_cache, 4, dims, strides, box)) != WPP_OK) return rc;
        if ((rc = make_map(ctx, &tv, v_cache, 4, dims, strides, box)) != WPP_OK) return rc;
    }

    wpp::SmallAttnParams p;
    memset(&p, 0, sizeof(p));
    p.plan = plan_dev;
    p.block_tables = block_tables;
    p.prefix_lens = prefix_lens;
    p.chunk_lens = chunk_lens;
    p.out = static_cast<__nv_bfloat16*>(out);
    p.lse = lse_or_null;
    p.tile_counter = static_cast<uint32_t*>(workspace);
    p.ws_o = reinterpret_cast<float*>(static_cast<char*>(workspace) + WPP_WS_HEADER_BYTES);
    p.ws_lse = p.ws_o + (size_t)hd->num_split_slots * 2 * WPP_HALF_M * d.head_dim;
    p.status = status_dev;
    p.o_token_stride = d.o_token_stride;
    p.o_head_stride = d.o_head_stride;
    p.num_q_heads = d.num_q_heads;
    p.group = d.num_q_heads / d.num_kv_heads;
    p.page_size = d.page_size;
    p.max_blocks = d.max_blocks_per_req;
    p.num_pages = d.num_pages;
    const double scale = d.sm_scale > 0.f ? (double)d.sm_scale : 1.0 / sqrt((double)d.head_dim);
    p.scale_log2 = (float)(scale * 1.4426950408889634);

    p.off_q_offsets = hd->off_q_offsets;
    p.off_prefix = hd->off_prefix;
    p.off_units = hd->off_units;
    p.num_units = hd->num_units;
    // The counter the CTAs take their tiles from starts at zero (a memset node on the caller's stream).  The small shape
    // needs none when its items are dealt out, the SM-wide one when every tile has a CTA: then nothing stands between the
    // kernel and the one before it.  SM-wide attention call of 2 x 4 tokens, us, with the memset and counters added on the
    // host's side of the bus 21.0, without the latter 16.6, without either 15.3.
    int e = 0;
    p.item_shift = hd->nonempty_halves > hd->num_units ? 1 : 0;
    const int64_t items = (int64_t)hd->num_units << p.item_shift;
    const int num_ctas = hd->shape == 2 ? (int)(items < hd->num_ctas ? items : hd->num_ctas) : hd->num_ctas;
    if (hd->shape == 2 ? hd->deal_items != 0 : hd->num_units <= num_ctas) {
        p.tile_counter = nullptr;
    } else {
        e = (int)cudaMemsetAsync(workspace, 0, WPP_WS_HEADER_BYTES, (cudaStream_t)cuda_stream);
        if (e != 0) return cuda_fail(ctx, e);
    }
    const int late = hd->shape == 2 ? 0 : choose_late_rescale(ctx, &p.totals);
    e = hd->shape == 2 ? wpp_launch_attention_small(d.head_dim, tq, &tk, &tv, &p, num_ctas, cuda_stream)
                       : wpp_launch_attention(d.head_dim, tq, &tk, &tv, &p, num_ctas, late, cuda_stream);
    if (e != 0) return cuda_fail(ctx, e);
    const_cast<wpp_ctx*>(ctx)->launches += 1;
    if (hd->num_combine > 0) {
        wpp::CombineParams c;
        memset(&c, 0, sizeof(c));
        c.plan = plan_dev;
        c.ws_o = p.ws_o;
        c.ws_lse = p.ws_lse;
        c.out = p.out;
        c.lse = lse_or_null;
        c.o_token_stride = d.o_token_stride;
        c.o_head_stride = d.o_head_stride;
        c.num_q_heads = d.num_q_heads;
        c.head_dim = d.head_dim;
        c.max_rows = hd->max_combine_rows;
        c.off_q_offsets = hd->off_q_offsets;
        c.off_combine = hd->off_combine;
        e = wpp_launch_combine(&c, hd->num_combine, cuda_stream);
        if (e != 0) return cuda_fail(ctx, e);
        const_cast<wpp_ctx*>(ctx)->launches += 1;
    }
    return WPP_OK;
}

// ---------------------------------------------------------------------------------------------------------------
// Entry point that allocates nothing: the tile counter and the split-KV partials live in the built-in scratch array
// whose address wpp_create looked up.
extern "C" int wpp_prefill_attention_varlen_static(const wpp_ctx* ctx, const wpp_batch_desc* desc, const void* q,
                                                   void* out, float* lse_or_null, const void* k_cache,
                                                   const void* v_cache, const int32_t* block_tables,
                                                   const int32_t* prefix_lens, const int32_t* chunk_lens,
                                                   const void* plan_host, const void* plan_dev, int32_t* status_dev,
                                                   void* cuda_stream) {
    if (!ctx || !ctx->static_scratch) return WPP_ERR_INVALID_ARG;
    wpp_batch_desc d;
    int rc = wpp_resolve_desc(desc, &d);
    if (rc != WPP_OK) return rc;
    const WppPlanHeader* hd = nullptr;
    if ((rc = wpp_check_plan(plan_host, &d, &hd)) != WPP_OK) return rc;
    if (hd->workspace_bytes > (uint64_t)WPP_STATIC_SCRATCH_BYTES) return WPP_ERR_WORKSPACE_TOO_SMALL;
    return wpp_prefill_attention_varlen(ctx, desc, q, out, lse_or_null, k_cache, v_cache, block_tables, prefix_lens,
                                        chunk_lens, plan_host, plan_dev, ctx->static_scratch,
                                        (size_t)WPP_STATIC_SCRATCH_BYTES, status_dev, cuda_stream);
}

// ---------------------------------------------------------------------------------------------------------------
// Recurrent-state layer.  Workspace of the chunk-parallel form's two passes: block offsets, then per (block, head) the cut mask,
// the decay products at sub-block ends and the ten operand arrays the preparation kernel leaves for the chain kernel.
struct KdaWorkspace {
    int64_t max_blocks, n_bh;
    size_t off_blk, off_mask, off_e, off_u0, off_op[6], off_sq[2], bytes;
};
static size_t up1k(size_t x) { return (x + 1023) / 1024 * 1024; }
static KdaWorkspace kda_workspace(const wpp_kda_desc* d) {
    KdaWorkspace w;
    w.max_blocks = d->total_tokens / 64 + 2 * (int64_t)d->num_requests;      // a chunk of C tokens touches <= C/64 + 2 blocks
    w.n_bh = w.max_blocks * d->num_heads;
    size_t off = 0;
    w.off_blk = off;  off += up1k(sizeof(int32_t) * ((size_t)d->num_requests + 1));
    w.off_mask = off; off += up1k(sizeof(uint64_t) * (size_t)w.n_bh);
    w.off_e = off;    off += up1k(sizeof(float) * (size_t)w.n_bh * 64 * 128);
    w.off_u0 = off;   off += up1k(sizeof(float) * (size_t)w.n_bh * 64 * 128);
    for (int i = 0; i < 6; ++i) { w.off_op[i] = off; off += up1k(2 * (size_t)w.n_bh * 64 * 128); }
    for (int i = 0; i < 2; ++i) { w.off_sq[i] = off; off += up1k(2 * (size_t)w.n_bh * 64 * 64); }
    w.bytes = off;
    return w;
}
static bool kda_desc_ok(const wpp_kda_desc* desc) {
    return desc && desc->num_requests >= 0 && desc->num_heads >= 1 && desc->num_slots >= 0 && desc->snap_interval >= 0 &&
           desc->max_snaps >= 0 && desc->total_tokens >= 0 && desc->layout >= 0 && desc->layout <= 3;
}

extern "C" size_t wpp_kda_workspace_bytes(const wpp_kda_desc* desc) {
    if (!kda_desc_ok(desc)) return 0;
    return kda_workspace(desc).bytes;
}

// Microseconds of the two passes over C tokens per request, measured on 148 SMs: preparation of a token of a chain on all SMs,
// a token of a chain that has an SM to itself, and what a token's operands take at the memory's rate.
constexpr double kPrepUs = 0.9e-3, kChainUs = 0.0525, kOperandsUs = 0.49e-3, kSegmentUs = 12.0;
struct KdaRates {
    double chains, tokens, prep, operands, chain;          // tokens: per request; us: on all SMs, of all chains
    double growth;                                         // what a chain takes over the preparation beside it; 0: no SMs for that
    KdaRates(const wpp_kda_desc* d, int sms) {
        chains = (double)d->num_requests * d->num_heads;
        tokens = (double)d->total_tokens / d->num_requests;
        prep = chains * tokens * kPrepUs * 148 / sms;
        operands = chains * tokens * kOperandsUs;
        chain = ceil(chains / sms) * tokens * kChainUs;
        growth = 2 * chains <= sms && tokens > 0 ? chain / (prep * sms / (sms - chains)) : 0.0;
    }
};

// Segments of the two-pass form.  Few long chains leave most SMs idle: the chunk is cut so that a segment's preparation runs
// beside the chain of the segment before.  A preparation takes whole rounds of items on its CTAs (two per SM; kRoundUs each
// on all SMs, kBesideUs beside a chain) and a start; a segment has as many rounds as fit beside the chain before it, so that
// only the first segment's preparation is waited for, and the last segment takes the rest.  Numbers of segments and of the first
// one's rounds (up to eight each of them, then in steps of a quarter) are those with the smallest total: the longer the chunk and
// the more chains, the more of both, so that no long preparation is left to the last segment; or segments that grow by the ratio of
// the two rates, where whole rounds do not come out (31 heads x 2,900 tokens).  Returns the number of segments and where they
// begin, in blocks; *us: the total.
// 1 x 16,384 tokens x 32 heads, us: in one piece 1,340, 4 equal segments 1,060, six that grow by the ratio of the two rates from
// 14 blocks on 1,084 (every chain but the last was done 20 to 37 us before the preparation beside it), so, five from 37 blocks on,
// 1,024 with no chain waiting; 1 x 8,192 584 | 556, 1 x 4,096 320 | 305, 1 x 2,048 189 | 178, 1 x 12,000 x 16 heads 738 | 701.
// Six growing segments | at most eight, the first of eight rounds at most | so: 1 x 65,536 x 32 heads 3,775 | 3,727 | 3,727,
// 98,304 5,577 | 6,174 | 5,486, 131,072 7,338 | 9,018 | 7,279, 65,536 x 36 3,889 | 4,973 | 3,889, 32,768 x 40 2,140 | 2,589 | 2,127,
// 2,900 x 31 236 | 244 | 236.
// Each segment beyond the eighth has to gain kMoreUs: it takes longer than by this count, 1 x 98,304 x 24 heads with nine 5,453, with
// eight 5,432, and 65,536 x 32 with eleven 3,733, where the count has gains of 6 and 18 us.
constexpr int kMaxSegments = 16;
constexpr double kRoundUs = 18.0, kBesideUs = 20.0, kStartUs = 6.0, kMoreUs = 8.0;
constexpr double kGapUs = 12.0;         // from a chain's last step to the next one's first
static int kda_segments(const wpp_kda_desc* d, int sms, double* us, int32_t* begin) {
    const KdaRates w(d, sms);
    const int64_t blocks = d->total_tokens / d->num_requests / 64 + 1;
    const double n = w.chains, step = 64 * kChainUs, all = 2.0 * sms, beside = 2.0 * (sms - n);
    double best_us = ceil((double)blocks * n / all) * kRoundUs + ceil(n / sms) * (double)blocks * step;
    begin[0] = 0;
    *us = best_us;
    if (w.growth <= 1.05) return 1;
    // of the segment behind one of `len` blocks: how many it has (two at least: it leaves its state in their operands' place), ...
    auto behind = [&](int64_t len) {
        const double fit = floor(((double)len * step + kGapUs - kStartUs) / kBesideUs);
        return (int64_t)fmax(2.0, floor(fmax(fit, 1.0) * beside / n));
    };
    // ... and from the start of the chain of `before` blocks to that of its own, if it has `len`
    auto wait = [&](int64_t len, int64_t before) {
        return fmax(ceil((double)len * n / beside) * kBesideUs + kStartUs, (double)before * step + kGapUs);
    };
    int best = 1;
    int64_t best_first = 0;
    for (int64_t rounds = 1; (double)rounds * all < (double)blocks * n; rounds += rounds < 8 ? 1 : rounds / 4) {
        const int64_t first = (int64_t)((double)rounds * all / n);
        double t = (double)rounds * kRoundUs;              // up to the start of the chain of the last segment so far
        int64_t len = first, done = first;
        for (int s = 2; s <= kMaxSegments && done < blocks; ++s) {
            const double rest = (double)(blocks - done), more = s > 8 ? kMoreUs * (s - 8) : 0.0;
            const double total = t + wait(blocks - done, len) + rest * step + more;
            if (total < best_us) { best_us = total; best = s; best_first = first; }
            const int64_t next = behind(len);
            t += wait(next, len);
            len = next;
            done += next;
        }
    }
    int64_t len = best_first;
    for (int s = 1; s < best; ++s, len = behind(len)) begin[s] = begin[s - 1] + (int32_t)len;
    for (int s = 2; s <= 6; ++s) {                         // segments that grow by the ratio of the two rates
        const double g = fmin(w.growth, 4.0), one = (double)blocks * (g - 1.0) / (pow(g, s) - 1.0);
        if (one < 4.0) break;
        int32_t at[7] = {0};
        double t = ceil(floor(one) * n / all) * kRoundUs;
        for (int i = 1; i <= s; ++i) {
            at[i] = i < s ? (int32_t)(one * (pow(g, i) - 1.0) / (g - 1.0)) : (int32_t)blocks;
            if (i > 1) t += wait(at[i] - at[i - 1], at[i - 1] - at[i - 2]);
        }
        t += (double)(at[s] - at[s - 1]) * step;
        if (t < best_us) {
            best_us = t;
            best = s;
            for (int i = 0; i < s; ++i) begin[i] = at[i];
        }
    }
    *us = best_us;
    return best;
}

// What the choice between the forms takes for the time of the two passes, without their launches: one piece, or the preparation of
// the first of a few growing segments and the chains.  Apart from kda_segments' total, which is for comparing cuts with one
// another: with one constant for the launches, this meets the measured times on either side of where the forms cross (us, this
// and 35 | two passes | group form: 1 x 2,048 x 32 heads 179 | 178 | 186, 2,048 x 24 169 | 168 | 185, 1,024 x 16 104 | 87 | 96; two
// chunks of 2,048 x 32 260 | 259) and stays within 5 % of them behind it (1 x 4,096 x 32 300 | 305, 16,384 982 | 1,024, 131,072
// 7,192 | 7,279).
static double kda_two_passes_us(const wpp_kda_desc* d, int sms) {
    const KdaRates w(d, sms);
    const double blocks = (double)(d->total_tokens / d->num_requests / 64 + 1), g = w.growth < 4.0 ? w.growth : 4.0;
    double us = w.prep + (w.chain > w.operands ? w.chain : w.operands);
    for (int s = 2; w.growth > 1.05 && s <= 6; ++s) {
        const double first = (g - 1.0) / (pow(g, s) - 1.0);
        if (first * blocks < 4.0) break;
        us = fmin(us, w.prep * first + w.chain + kSegmentUs * (s - 1));
    }
    return us;
}

// Which chunk-parallel kernel: 0 = blocks of 64 tokens in two passes (preparation for all blocks in parallel, then the
// chain), 1..3 = groups of 16 tokens with the state in registers (wpp_kda_group.cu), in CTAs of 128, 64 or 32 columns.
// The two-pass form reads and writes 144 KB of operands per block but its chain is the fastest per token; the group form
// has nothing in front of its chain and moves nothing but inputs and outputs.  The estimates below are microseconds for
// C tokens per request, measured on 148 SMs (us; group with 128 / 64 / 32 columns | two passes):
//     requests x heads x tokens    8x32x2048  669 / 853 / 1285 | 744     1x32x512    93 /  77 /   56 |   71
//                                  4x32x256    56 /  67 /  116 |  79     1x8x2048   333 / 273 /  188 |  153
//                                  4x32x4096  661 / 857 / 1443 | 732     2x32x2048  335 / 280 /  378 |  259
//                                  8x32x64     42 /  44 /   75 |  58     64x32x256  652 / 775 / 1469 |  798
// Error against 64 bits, rms of the states over their rms, 8 x 2,048 tokens x 32 heads: 4.35e-6 (two passes: 5.09e-6); outputs
// 1.6595e-3 for both, the rounding to bf16.
//
// These are waves of equal chunks, and a wave lasts at least as long as its longest chain, which costs three times as much per
// token here as in the two passes.  The lengths are on the device: the group form's CTAs look at them, and a wave with a chunk
// longer than *longest is left to the two passes queued behind (which end at once if it is not).  For whole chains *longest is the
// length up to which the group form is the faster one however the rest is distributed: no order of its CTAs takes longer than
// its rounds all of the longest chunk, nor than the chunks spread evenly and the longest on top; the two passes are taken for
// equal chunks, where they are fastest.  us, two passes | group form whatever the lengths | now:
//     8 x 32 heads, 14,000 and 7 x 340 tokens 1261 | 2108 | 1263     8 x 32, 8,192 and 7 x 1,170 960 | 1248 | 959
//     9 x 8 heads, 16,000 and 8 x 48 tokens 1004 | 2055 | 1004        4 x 32, 512 and 3 x 64 85 | 92 | 83
// For cut chains *longest is an estimate and no bound: an even spread with half of the longest piece on top, or the longest chain
// alone.  It leaves out that waiting pieces hold an SM and that several chunks may have that length: 7 x 1,590 and 9 x 8 tokens
// (32 heads), just not too long for 2 pieces, two passes | cut 554 | 550, 4 x 1,000 and 2 x 2,330 476 | 450, 8 x 1,024..2,048
// 537 | 480.
// What it costs to ask: the empty launches behind a wave of equal chunks (whole chains) 8 x 2,048 669 -> 676, 4 x 256 56 -> 64,
// 8 x 64 42 -> 50, 64 x 256 652 -> 673; the group kernel's empty CTAs, one per piece, in front of a wave that is then left to the
// two passes, 1 to 4 us (1,290 + 3 x 60 + 40 tokens 151 -> 152, 11 x 1..433 210 -> 214, 20 x 1..524 (8 heads) 111 -> 113).
constexpr double kGroupUs = 12.0;       // what a launch takes before and after its chains
constexpr double kPieceUs = 8.0;        // what a piece of a chain takes besides its tokens (6 measured: not cut where it hardly gains)
constexpr double kPieceTokens = 96.0;   // tokens that a piece has at least, on average
constexpr int kMaxPieces = 8;
// Pieces per chain of the 128-column CTAs, one CTA per SM: whole chains leave the last of few rounds partly empty (256 chains on
// 148 SMs take two rounds of which the second is 73 % full).  A piece of a chain waits for the one before, which started a
// whole round of chains earlier: only with at least as many chains as SMs.  Measured, us, in 1 / 2 / 4 / 5 / 8 pieces (32 heads):
// 8 x 2,048 672 / 693 / 637 / 666 / 683, 8 x 1,024 350 / 369 / 352 / 371 / 398, 5 x 1,000 345 / 279 / 250 / 249 / 257,
// 6 x 2,048 670 / 528 / 542 / 520 / 531 (3 pieces: 479), 64 x 256 667 / 787 / 988: cut where it gives 3 % by this estimate.
// It takes all chunks for equally long.  Where some are far shorter, the long chains alone may fit the SMs at once, and short
// pieces cost more than they even out: 4 x 166 and 22 tokens whole 45 us, in 2 pieces 53 (equal chunks, 5 x 160: 72 | 70).
// Hence kPieceTokens: what shorter pieces would gain on equal chunks is 3 to 4 %, 5 x 200 tokens 86 | 82.
static int kda_pieces(double n, double C, int sms, double us_per_token, double* us) {
    int best = 1;
    double best_us = ceil(n / sms) * C * us_per_token;
    const double whole = best_us + ceil(n / sms) * kPieceUs;
    double least = 0.97 * whole;
    for (int k = 2; k <= kMaxPieces && n >= sms && C >= kPieceTokens * k; ++k) {
        const double t = ceil(n * k / sms) * (C / k * us_per_token + kPieceUs);
        if (t < least) { best = k; least = t; best_us = t - ceil(n / sms) * kPieceUs; }
    }
    *us = best_us;
    return best;
}
static int kda_chunk_form(const wpp_kda_desc* d, int sms, int64_t* longest, int* pieces) {
    const double n = (double)d->num_requests * d->num_heads, C = (double)d->total_tokens / d->num_requests;
    const double two_passes = kda_two_passes_us(d, sms) + 35.0;
    const struct { double ctas, at_once, us_per_token; } form[4] = {{},
                                                                    {n, (double)sms, 0.165},                                 // one CTA per SM
                                                                    {2 * n, 2.0 * sms, 2 * n <= sms ? 0.14 : 0.2},           // two per SM
                                                                    {4 * n, (double)sms, 0.088}};
    int best = 0;
    double best_us = two_passes;
    double whole_us = 0.0;                  // form 1 with its chains cut
    *pieces = kda_pieces(n, C, sms, form[1].us_per_token, &whole_us);
    for (int i = 1; i < 4; ++i) {
        const double us = i == 1 ? whole_us : ceil(form[i].ctas / form[i].at_once) * C * form[i].us_per_token;
        if (us < best_us) { best = i; best_us = us; }
    }
    if (best > 0) {
        const double per_token = form[best].us_per_token, budget = two_passes - kGroupUs;
        double all_longest, spread;
        if (best == 1 && *pieces > 1) {
            // cut chains: the wave is done when the longest is, or when the SMs are through with everything and half a piece
            const double k = *pieces, work = n * C / sms * per_token + ceil(n * k / sms) * kPieceUs;
            all_longest = C * budget / whole_us;
            spread = (budget - work) * 2.0 * k / per_token;
            const double alone = (budget - k * kPieceUs) / per_token;
            if (alone < spread) spread = alone;
        } else {
            all_longest = budget / per_token / ceil(form[best].ctas / form[best].at_once);
            spread = budget / per_token - form[best].ctas * C / form[best].at_once;
        }
        *longest = (int64_t)(all_longest > spread ? all_longest : spread);
        if (d->num_requests > 1 && (double)*longest < C) best = 0;
    }
    return best;
}
// (the choices by themselves, for the tests: no GPU needed)
extern "C" int wpp_kda_choice(const wpp_kda_desc* d, int sms, int64_t* longest, int* pieces) {
    if (!kda_desc_ok(d) || d->num_requests < 1 || d->total_tokens < 64 * (int64_t)d->num_requests || sms < 1) return -1;
    *longest = 0;
    const int form = kda_chunk_form(d, sms, longest, pieces);
    if (form != 1) *pieces = 1;
    return form;
}
extern "C" int wpp_kda_cut(const wpp_kda_desc* d, int sms, double* us, int32_t* begin /* [16] */) {
    if (!kda_desc_ok(d) || d->num_requests < 1 || sms < 1) return -1;
    return kda_segments(d, sms, us, begin);
}

extern "C" int wpp_kda_chunk(const wpp_ctx* ctx, const wpp_kda_desc* desc, const void* q, const void* k, const void* v,
                             const float* alpha, const float* beta, const int64_t* row_offsets,
                             const int32_t* prefix_lens, float* state_pool, const int32_t* state_in,
                             const int32_t* state_out, const int32_t* snap_slots, void* out, void* workspace,
                             size_t workspace_bytes, int32_t* status_dev, void* cuda_stream) {
    if (!ctx || !kda_desc_ok(desc)) return WPP_ERR_INVALID_ARG;
    if (desc->d_k != 128 || desc->d_v != 128) return WPP_ERR_UNSUPPORTED;
    if (desc->num_requests > 65535) return WPP_ERR_UNSUPPORTED;      // one grid row per request
    if (desc->num_requests == 0) return WPP_OK;
    if (int rc = wpp_ctx_check_device(ctx)) return rc;
    if (!row_offsets || !state_in || !state_out) return WPP_ERR_INVALID_ARG;
    if (desc->num_slots > 0 && !state_pool) return WPP_ERR_INVALID_ARG;
    if (desc->total_tokens > 0 && (!q || !k || !v || !alpha || !beta || !out)) return WPP_ERR_INVALID_ARG;
    if (desc->snap_interval > 0 && !prefix_lens) return WPP_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(alpha) || !aligned16(out) || !aligned16(state_pool))
        return WPP_ERR_INVALID_ARG;
    // Which form: the chunk-parallel tensor-core form needs a workspace and pays off from about a block of tokens
    // per request; the token-by-token forms need none.
    const KdaWorkspace w = kda_workspace(desc);
    bool tensor_form = desc->layout == 3;
    if (desc->layout == 0)
        tensor_form = workspace && workspace_bytes >= w.bytes && desc->total_tokens >= 64 * (int64_t)desc->num_requests;
    if (tensor_form) {
        if (!workspace || workspace_bytes < w.bytes) return WPP_ERR_WORKSPACE_TOO_SMALL;
        if ((reinterpret_cast<uintptr_t>(workspace) & 255) != 0) return WPP_ERR_INVALID_ARG;
        if (w.n_bh * 64 > 0x7fffffffll || desc->total_tokens > 0x7fffffffll) return WPP_ERR_UNSUPPORTED;
    }
    // (layout 3 is always the two passes: their result does not depend on how long the rest of the chunk is)
    int64_t longest = 0;
    int pieces = 1;
    const int form = tensor_form && desc->layout == 0 ? kda_chunk_form(desc, ctx->sm_count, &longest, &pieces) : 0;
    // a single chunk's length is known here: nothing has to stand behind the group form
    const bool gated = form > 0 && desc->num_requests > 1;
    int e;
    if (!tensor_form || form > 0) {
        wpp::KdaGroupParams p;
        memset(&p, 0, sizeof(p));
        p.q = static_cast<const __nv_bfloat16*>(q);
        p.k = static_cast<const __nv_bfloat16*>(k);
        p.v = static_cast<const __nv_bfloat16*>(v);
        p.alpha = alpha;
        p.beta = beta;
        p.row_offsets = row_offsets;
        p.prefix_lens = prefix_lens;
        p.state_pool = state_pool;
        p.state_in = state_in;
        p.state_out = state_out;
        p.snap_slots = desc->max_snaps > 0 ? snap_slots : nullptr;
        p.out = static_cast<__nv_bfloat16*>(out);
        p.status = status_dev;
        p.num_requests = desc->num_requests;
        p.num_heads = desc->num_heads;
        p.num_slots = desc->num_slots;
        p.snap_interval = desc->snap_interval;
        p.max_snaps = desc->max_snaps;
        if (tensor_form) {
            p.longest = longest;
            p.pieces = form == 1 ? pieces : 1;
            p.hand = reinterpret_cast<float4*>(static_cast<char*>(workspace) + w.off_e);              // (n_bh >= 2 R H rows of 32 KB)
            p.ticket = reinterpret_cast<int32_t*>(static_cast<char*>(workspace) + w.off_u0);
            p.hand_seen = p.ticket + 1;
            p.blk_off = gated ? reinterpret_cast<int32_t*>(static_cast<char*>(workspace) + w.off_blk) : nullptr;
            CUtensorMap maps[4];
            memset(maps, 0, sizeof(maps));
            int rc;
            if (desc->total_tokens > 0) {
                // boxes of the 16 rows of a group: whole rows of q, k and alpha (fp32 as a bf16 map with twice the elements:
                // the copies move bytes), 64-column swizzled halves of v
                const uint64_t H = (uint64_t)desc->num_heads, T = (uint64_t)desc->total_tokens;
                const uint64_t dims[3] = {128, H, T}, dims_a[3] = {256, H, T};
                const uint64_t strides[2] = {256, 256 * H}, strides_a[2] = {512, 512 * H};
                const uint32_t box[3] = {128, 1, 16}, box_v[3] = {64, 1, 16}, box_a[3] = {256, 1, 16};
                if ((rc = make_map(ctx, &maps[0], q, 3, dims, strides, box, false)) != WPP_OK) return rc;
                if ((rc = make_map(ctx, &maps[1], k, 3, dims, strides, box, false)) != WPP_OK) return rc;
                if ((rc = make_map(ctx, &maps[2], v, 3, dims, strides, box_v)) != WPP_OK) return rc;
                if ((rc = make_map(ctx, &maps[3], alpha, 3, dims_a, strides_a, box_a, false)) != WPP_OK) return rc;
            }
            e = wpp_launch_kda_group(&p, maps, form, cuda_stream);
        } else {
            e = wpp_launch_kda(&p, ctx->sm_count, desc->layout, cuda_stream);
        }
        if (e != 0) return cuda_fail(ctx, e);
        const_cast<wpp_ctx*>(ctx)->launches += 1;
    }
    if (tensor_form && (form == 0 || gated)) {
        char* ws = static_cast<char*>(workspace);
        wpp::KdaTcParams p;
        memset(&p, 0, sizeof(p));
        p.q = static_cast<const __nv_bfloat16*>(q);
        p.k = static_cast<const __nv_bfloat16*>(k);
        p.v = static_cast<const __nv_bfloat16*>(v);
        p.alpha = alpha;
        p.beta = beta;
        p.row_offsets = row_offsets;
        p.prefix_lens = prefix_lens;
        p.state_pool = state_pool;
        p.state_in = state_in;
        p.state_out = state_out;
        p.snap_slots = desc->max_snaps > 0 ? snap_slots : nullptr;
        p.out = static_cast<__nv_bfloat16*>(out);
        p.status = status_dev;
        p.num_requests = desc->num_requests;
        p.num_heads = desc->num_heads;
        p.num_slots = desc->num_slots;
        p.snap_interval = desc->snap_interval;
        p.max_snaps = desc->max_snaps;
        p.blk_off = reinterpret_cast<int32_t*>(ws + w.off_blk);
        p.ws_mask = reinterpret_cast<unsigned long long*>(ws + w.off_mask);
        p.ws_e = reinterpret_cast<float*>(ws + w.off_e);
        p.ws_u0 = reinterpret_cast<float*>(ws + w.off_u0);
        __nv_bfloat16** ops[6] = {&p.ws_w0_h, &p.ws_w0_l, &p.ws_qt_h, &p.ws_qt_l, &p.ws_kb_h, &p.ws_kb_l};
        __nv_bfloat16** sqs[2] = {&p.ws_m_h, &p.ws_m_l};
        CUtensorMap maps[13];
        int rc;
        for (int i = 0; i < 6; ++i) {
            *ops[i] = reinterpret_cast<__nv_bfloat16*>(ws + w.off_op[i]);
            const uint64_t dims[2] = {128, (uint64_t)w.n_bh * 64};
            const uint64_t strides[1] = {256};
            const uint32_t box[2] = {64, 64};
            if ((rc = make_map(ctx, &maps[i], *ops[i], 2, dims, strides, box)) != WPP_OK) return rc;
        }
        for (int i = 0; i < 2; ++i) {
            *sqs[i] = reinterpret_cast<__nv_bfloat16*>(ws + w.off_sq[i]);
            const uint64_t dims[2] = {64, (uint64_t)w.n_bh * 64};
            const uint64_t strides[1] = {128};
            const uint32_t box[2] = {64, 64};
            if ((rc = make_map(ctx, &maps[6 + i], *sqs[i], 2, dims, strides, box)) != WPP_OK) return rc;
        }
        // fp32 arrays (U0, alpha) as bf16 maps with twice the elements per row: the copies move bytes
        {
            const uint64_t dims[2] = {256, (uint64_t)w.n_bh * 64};
            const uint64_t strides[1] = {512};
            const uint32_t box[2] = {64, 64};
            if ((rc = make_map(ctx, &maps[8], p.ws_u0, 2, dims, strides, box)) != WPP_OK) return rc;
        }
        if (desc->total_tokens > 0) {
            const uint64_t H = (uint64_t)desc->num_heads, T = (uint64_t)desc->total_tokens;
            const void* in[3] = {q, k, v};
            const uint32_t box[3] = {64, 1, 64};
            for (int i = 0; i < 3; ++i) {
                const uint64_t dims[3] = {128, H, T};
                const uint64_t strides[2] = {256, 256 * H};
                if ((rc = make_map(ctx, &maps[9 + i], in[i], 3, dims, strides, box)) != WPP_OK) return rc;
            }
            const uint64_t dims[3] = {256, H, T};
            const uint64_t strides[2] = {512, 512 * H};
            if ((rc = make_map(ctx, &maps[12], alpha, 3, dims, strides, box)) != WPP_OK) return rc;
        }
        // few long chains leave most SMs to the next segment's preparation (not behind the group form: each segment is two
        // launches that usually have nothing to do)
        p.gated = gated;
        int32_t seg_begin[kMaxSegments] = {0};
        double us = 0.0;
        const int segments = gated ? 1 : kda_segments(desc, ctx->sm_count, &us, seg_begin);
        e = wpp_launch_kda_tc(&p, maps, desc->total_tokens > 0 ? (int)w.max_blocks : 0, ctx->sm_count, segments, seg_begin,
                              cuda_stream);
        if (e != 0) return cuda_fail(ctx, e);
        const_cast<wpp_ctx*>(ctx)->launches += (gated ? 0 : 1) + 2 * segments;
    }
    return WPP_OK;
}
