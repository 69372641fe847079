// Prefix hints (Section 4.3): chained hashes of full token blocks (GPU and host) and the counted, sharded index
// with the gallop-and-bisect probe (host).
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <new>
#include <unordered_map>

#include "../../include/wpp.h"
#include "wpp_host.h"

namespace {

__host__ __device__ inline uint64_t mix64(uint64_t x) {     // splitmix64 finaliser
    x ^= x >> 30;
    x *= 0xBF58476D1CE4E5B9ull;
    x ^= x >> 27;
    x *= 0x94D049BB133111EBull;
    x ^= x >> 31;
    return x;
}
__host__ __device__ inline uint64_t token_term(int32_t token, uint32_t k) {
    return mix64((((uint64_t)(uint32_t)token << 32) | k) ^ 0xD6E8FEB86659FD93ull);
}
__host__ __device__ inline uint64_t chain_step(uint64_t parent, uint64_t digest, uint64_t extra, uint64_t salt_term) {
    return mix64(parent ^ mix64(digest + extra) ^ salt_term);
}

// Digests.  A warp takes kBlocks consecutive blocks: 16 or 8 token loads are in flight together, and the request the
// blocks start in is found once, by a search whose every step is one load of 32 offsets (a bisection by one lane per
// block was eight dependent loads in front of every block).  Every warp has one job, so that the hardware's own
// scheduling of CTAs covers one warp's search with another's arithmetic.  What is left where a block's hash will go is
// c ^ c >> 30 with c = mix64(digest + extraKeys) ^ salt term: everything of the chain step that does not depend on the
// parent hash.  Bound by the arithmetic of the terms (two 64-bit products per token).
template <int kBlocks>
__global__ void __launch_bounds__(256) wpp_block_digest_kernel(const int32_t* __restrict__ tokens,
                                                                const int64_t* __restrict__ token_offsets,
                                                                const int64_t* __restrict__ block_offsets,
                                                                int num_requests, int block_size, uint64_t salt_term,
                                                                const uint64_t* __restrict__ extra,
                                                                uint64_t* __restrict__ out, int64_t total_blocks) {
    const int lane = threadIdx.x & 31;
    const int64_t first = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kBlocks;
    if (first >= total_blocks) return;
    int lo = 0, hi = num_requests;              // largest i with block_offsets[i] <= first
    while (hi - lo > 1) {
        const int width = (hi - lo + 31) / 32, i = lo + lane * width;
        const unsigned le = __ballot_sync(0xffffffffu, i < hi && block_offsets[i] <= first) | 1u;
        const int last = 31 - __clz((int)le);
        hi = min(hi, lo + (last + 1) * width);
        lo += last * width;
    }
    // lane j < kBlocks: where block first + j starts
    const int cnt = (int)min((int64_t)kBlocks, total_blocks - first);
    int64_t start = 0;
    if (lane < cnt) {
        int r = lo;
        while (r + 1 < num_requests && block_offsets[r + 1] <= first + lane) ++r;
        start = token_offsets[r] + (first + lane - block_offsets[r]) * block_size;
    }
    const int32_t* src[kBlocks];
    uint64_t d[kBlocks];
#pragma unroll
    for (int j = 0; j < kBlocks; ++j) {
        src[j] = tokens + __shfl_sync(0xffffffffu, start, j);
        d[j] = 0;
    }
    constexpr int kU = kBlocks == 1 ? 8 : 2;
    for (int k0 = 0; k0 < block_size; k0 += 32 * kU) {
        int32_t t[kBlocks][kU];
#pragma unroll
        for (int j = 0; j < kBlocks; ++j)
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int k = k0 + 32 * u + lane;
                t[j][u] = (j < cnt && k < block_size) ? __ldg(src[j] + k) : 0;
            }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int k = k0 + 32 * u + lane;
            if (k0 + 32 * u >= block_size) break;
#pragma unroll
            for (int j = 0; j < kBlocks; ++j) d[j] += k < block_size ? token_term(t[j][u], (uint32_t)k) : 0ull;
        }
    }
    uint64_t mine = 0;
#pragma unroll
    for (int j = 0; j < kBlocks; ++j) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d[j] += __shfl_xor_sync(0xffffffffu, d[j], o);
        if (lane == j) mine = d[j];
    }
    if (lane < cnt) {
        const uint64_t c = mix64(mine + (extra ? extra[first + lane] : 0ull)) ^ salt_term;
        out[first + lane] = c ^ (c >> 30);
    }
}

// The chain H_i = mix64(H_{i-1} ^ mix64(digest_i + extraKeys_i) ^ salt term) is sequential by definition: a
// warp walks a request's blocks, and what bounds it is the step's own dependent arithmetic.
// With z the value before mix64's last shift, h = z ^ z >> 31, the next step starts from
//     h ^ c ^ (h ^ c) >> 30  =  z ^ z >> 30 ^ z >> 31 ^ z >> 61 ^ (c ^ c >> 30),
// whose shifts are independent of one another and whose last term the digests left ready: two dependent operations
// between the multiplications instead of four.  The step works on 32-bit halves, because a 64-bit product's low half is
// there long before its high half: all of a shift that comes from the low half is folded in while the high half is on its
// way, and the high half is the sum of three products that do not wait for one another.  Its shifts and exclusive ors are
// issued every other clock at most, so their number counts as well: one funnel shift takes what z >> 30 needs of both
// halves, and z ^ z >> 31, the hash itself, is left to whoever stores it.  64 requests x 3,125 blocks, the fused kernel with
// its tokens in L2: 64-bit operations 143 us, halves with wide products 129, in this order 127.5, with the funnel shift, the
// hash left out and four steps a turn 117 (69 clocks a step; eight steps a turn 123, two 126, the same without the funnel
// shift 123).
// The warp moves kStage blocks at a time through shared memory - the next
// stage's loads are in flight while this one is chained, the finished hashes leave as coalesced stores - so that the
// walk never waits on global memory; inside a stage a turn's terms are read a turn ahead and its results written after its
// steps (a load that may alias the store before it would put shared-memory latency into every step).  All lanes walk alike:
// one lane alone takes 1 % longer.
__device__ __forceinline__ uint32_t xor3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0x96;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
__device__ __forceinline__ uint32_t mul_hi(uint32_t a, uint32_t b) {     // (apart from the low half: a wide product is later)
    uint32_t r;
    asm("mul.hi.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t mul_lo(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("mul.lo.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint64_t chain_product(uint64_t z, uint64_t c) {
    constexpr uint32_t k1l = 0x1CE4E5B9u, k1h = 0xBF58476Du, k2l = 0x133111EBu, k2h = 0x94D049BBu;
    const uint32_t l = (uint32_t)z, h = (uint32_t)(z >> 32), cl = (uint32_t)c, ch = (uint32_t)(c >> 32);
    const uint32_t early = xor3(l, cl, l >> 31);                               // ... ^ the low halves of z >> 61, 31 and 30
    const uint32_t xl = xor3(early, h >> 29, h << 1) ^ __funnelshift_l(l, h, 2), xh = xor3(h ^ ch, h >> 30, h >> 31);
    const uint32_t pl = mul_lo(xl, k1l), ph = mul_hi(xl, k1l) + mul_lo(xl, k1h) + mul_lo(xh, k1l);
    const uint32_t yl = xor3(pl, pl >> 27, ph << 5), yh = ph ^ (ph >> 27);
    const uint32_t ql = mul_lo(yl, k2l), qh = mul_hi(yl, k2l) + mul_lo(yl, k2h) + mul_lo(yh, k2l);
    return ((uint64_t)qh << 32) | ql;
}
__device__ __forceinline__ uint64_t chain_hash(uint64_t z) { return z ^ (z >> 31); }
// The steps of the terms m[0, cnt), whose products go to h; both have room for kMost values.  (Steps past the last term
// compute on values nobody reads.)
template <int kMost>
__device__ __forceinline__ void chain_steps(uint64_t& z, const uint64_t* m, uint64_t* h, int cnt) {
    constexpr int kTurn = 4;
    static_assert(kMost % kTurn == 0, "whole turns");
    uint64_t c[kTurn];
#pragma unroll
    for (int j = 0; j < kTurn; ++j) c[j] = m[j];
#pragma unroll 1
    for (int i = 0; i < cnt; i += kTurn) {
        uint64_t next[kTurn];                              // (past the last turn: the first one's again, not used)
        const int at = i + kTurn < kMost ? i + kTurn : 0;
#pragma unroll
        for (int j = 0; j < kTurn; ++j) next[j] = m[at + j];
#pragma unroll
        for (int j = 0; j < kTurn; ++j) c[j] = z = chain_product(z, c[j]);
#pragma unroll
        for (int j = 0; j < kTurn; ++j) h[i + j] = c[j];
#pragma unroll
        for (int j = 0; j < kTurn; ++j) c[j] = next[j];
    }
}
constexpr int kStage = 128, kPerLane = kStage / 32;
__global__ void __launch_bounds__(32) wpp_hash_chain_kernel(const int64_t* __restrict__ block_offsets,
                                                            uint64_t* __restrict__ hashes) {
    __shared__ uint64_t buf[kStage], done[kStage];
    const int lane = threadIdx.x;
    const int64_t b0 = block_offsets[blockIdx.x], n = block_offsets[blockIdx.x + 1] - b0;
    uint64_t* h = hashes + b0;
    uint64_t nxt[kPerLane];
#pragma unroll
    for (int u = 0; u < kPerLane; ++u) nxt[u] = u * 32 + lane < n ? h[u * 32 + lane] : 0ull;
    uint64_t z = 0;
    for (int64_t first = 0; first < n; first += kStage) {
#pragma unroll
        for (int u = 0; u < kPerLane; ++u) buf[u * 32 + lane] = nxt[u];
        __syncwarp();
#pragma unroll
        for (int u = 0; u < kPerLane; ++u) {
            const int64_t i = first + kStage + u * 32 + lane;
            nxt[u] = i < n ? h[i] : 0ull;
        }
        chain_steps<kStage>(z, buf, done, (int)min((int64_t)kStage, n - first));
        __syncwarp();
#pragma unroll
        for (int u = 0; u < kPerLane; ++u) {
            const int64_t i = first + u * 32 + lane;
            if (i < n) h[i] = chain_hash(done[u * 32 + lane]);
        }
        __syncwarp();
    }
}

// Digests and chain of long prompts in one kernel, a CTA per request: twelve warps work on the digests of the next stage of
// 96 blocks while one warp chains the current ones out of shared memory, so that only the first stage's digests stand in
// front of the chain.  The chain's warp is the only one of its scheduler (warps 7, 11 and 15 leave at once): beside digest
// warps its dependent steps waited for issue slots (170 us instead of 144 for 64 requests x 3,125 blocks of 64 tokens).
// The tokens of a stage are requested a stage ahead (requested with their use, a stage of tokens that come from HBM took
// longer than its chain: 154 us however short the chain's step), the chain's next terms a turn ahead.
constexpr int kFusedWarps = 12, kFusedStage = 8 * kFusedWarps, kFusedThreads = 512;
__global__ void __launch_bounds__(kFusedThreads, 1) wpp_hash_fused_kernel(const int32_t* __restrict__ tokens,
                                                                          const int64_t* __restrict__ token_offsets,
                                                                          const int64_t* __restrict__ block_offsets,
                                                                          int block_size, uint64_t salt_term,
                                                                          const uint64_t* __restrict__ extra,
                                                                          uint64_t* __restrict__ out) {
    __shared__ uint64_t s_m[2][kFusedStage], s_h[2][kFusedStage];
    const int req = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp > 3 && (warp & 3) == 3) return;
    const int dw = warp - (warp >> 2);                 // digest warps 0..11 (the chain's warp is 3)
    auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(32 * (kFusedWarps + 1)) : "memory"); };
    const int64_t b0 = block_offsets[req], n = block_offsets[req + 1] - b0;
    const int32_t* src = tokens + token_offsets[req];
    const int n_stages = (int)((n + kFusedStage - 1) / kFusedStage);
    int32_t t[8][2];                                   // the tokens of the warp's next eight blocks, on their way
    auto load = [&](int s) {
        const int64_t first = (int64_t)s * kFusedStage + dw * 8;
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = 32 * u + lane;
                t[j][u] = (k < block_size && first + j < n) ? __ldg(src + (first + j) * block_size + k) : 0;
            }
    };
    auto digest = [&](int s) {
        const int64_t first = (int64_t)s * kFusedStage + dw * 8;
        uint64_t d[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) d[j] = 0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int k = 32 * u + lane;
            if (32 * u >= block_size) break;
#pragma unroll
            for (int j = 0; j < 8; ++j) d[j] += k < block_size ? token_term(t[j][u], (uint32_t)k) : 0ull;
        }
        load(s + 1);
        // lane l ends with the sum of block l & 7: with every exchange it hands over the half of its blocks that it does not
        // keep (nine exchanges instead of forty; a stage's digests 4.0 K clocks instead of 4.9 K)
        const bool hi4 = lane & 4, hi2 = lane & 2, hi1 = lane & 1;
        uint64_t e4[4], e2[2];
#pragma unroll
        for (int j = 0; j < 4; ++j) e4[j] = (hi4 ? d[j + 4] : d[j]) + __shfl_xor_sync(0xffffffffu, hi4 ? d[j] : d[j + 4], 4);
#pragma unroll
        for (int j = 0; j < 2; ++j) e2[j] = (hi2 ? e4[j + 2] : e4[j]) + __shfl_xor_sync(0xffffffffu, hi2 ? e4[j] : e4[j + 2], 2);
        uint64_t mine = (hi1 ? e2[1] : e2[0]) + __shfl_xor_sync(0xffffffffu, hi1 ? e2[0] : e2[1], 1);
        mine += __shfl_xor_sync(0xffffffffu, mine, 8);
        mine += __shfl_xor_sync(0xffffffffu, mine, 16);
        if (lane < 8) {                     // (entries past the request's last block are never used)
            const uint64_t c = mix64(mine + ((extra && first + lane < n) ? extra[b0 + first + lane] : 0ull)) ^ salt_term;
            s_m[s & 1][dw * 8 + lane] = c ^ (c >> 30);
        }
    };
    if (warp != 3 && n_stages > 0) {
        load(0);
        digest(0);
    }
    sync();
    uint64_t z = 0;
    for (int s = 0; s <= n_stages; ++s) {
        if (warp == 3) {
            if (s < n_stages) chain_steps<kFusedStage>(z, s_m[s & 1], s_h[s & 1], (int)min((int64_t)kFusedStage, n - (int64_t)s * kFusedStage));
            __syncwarp();
        } else {
            if (s > 0) {
                const int64_t i = (int64_t)(s - 1) * kFusedStage + dw * 8 + lane;
                if (lane < 8 && i < n) out[b0 + i] = chain_hash(s_h[(s - 1) & 1][dw * 8 + lane]);
            }
            if (s + 1 < n_stages) digest(s + 1);
        }
        sync();
    }
}

constexpr int kShards = 16;
struct Key {
    int32_t window;
    uint64_t hash;
    bool operator==(const Key& o) const { return window == o.window && hash == o.hash; }
};
struct KeyHash {
    size_t operator()(const Key& k) const { return (size_t)mix64(k.hash ^ ((uint64_t)(uint32_t)k.window << 1)); }
};

}  // namespace

struct wpp_hint_index {
    std::unordered_map<Key, int64_t, KeyHash> map[kShards];
    mutable std::mutex lock[kShards];
    static int shard(uint64_t h) { return (int)((h >> 7) & (kShards - 1)); }
    bool has(int32_t window, uint64_t h) const {
        const int s = shard(h);
        std::lock_guard<std::mutex> g(lock[s]);
        return map[s].count(Key{window, h}) != 0;
    }
};

extern "C" int wpp_hash_blocks(const wpp_ctx* ctx, const int32_t* tokens, const int64_t* token_offsets,
                               const int64_t* block_offsets, int32_t num_requests, int32_t block_size, uint64_t salt,
                               const uint64_t* extra, uint64_t* hashes_out, int64_t total_blocks, void* cuda_stream) {
    if (!ctx || num_requests < 0 || block_size < 1 || total_blocks < 0) return WPP_ERR_INVALID_ARG;
    if (num_requests == 0 || total_blocks == 0) return WPP_OK;
    if (!tokens || !token_offsets || !block_offsets || !hashes_out) return WPP_ERR_INVALID_ARG;
    if (int rc = wpp_ctx_check_device(ctx)) return rc;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const uint64_t salt_term = salt * 0x9E3779B97F4A7C15ull;
    // One kernel when every request can have an SM and its twelve warps keep up with the chain (blocks of up to 64 tokens:
    // an SM makes a block's digest in less than a chain step).  us, one kernel | two, both before the chain's step was
    // shortened for both: 64 requests x 3,125 blocks of 64 144 | 172, 64 x 100 11 | 15, 148 x 3,125 156 | 222; blocks of 128:
    // 1 x 1,500 90 | 72, 64 x 3,125 269 | 199.
    const int sms = wpp_ctx_sm_count(ctx);
    if (num_requests <= sms && block_size <= 64) {
        wpp_hash_fused_kernel<<<(unsigned)num_requests, kFusedThreads, 0, st>>>(tokens, token_offsets, block_offsets, block_size,
                                                                               salt_term, extra, hashes_out);
        return cudaGetLastError() == cudaSuccess ? WPP_OK : WPP_ERR_CUDA;
    }
    // eight blocks per warp once that still gives every SM 32 warps; one below, where a warp's latency is all that counts
    const bool wide = total_blocks >= 8ll * 32 * sms;
    const int64_t ctas = (total_blocks + (wide ? 63 : 7)) / (wide ? 64 : 8);
    if (ctas > 0x7fffffffll) return WPP_ERR_INVALID_ARG;
    if (wide)
        wpp_block_digest_kernel<8><<<(unsigned)ctas, 256, 0, st>>>(tokens, token_offsets, block_offsets, num_requests,
                                                                   block_size, salt_term, extra, hashes_out, total_blocks);
    else
        wpp_block_digest_kernel<1><<<(unsigned)ctas, 256, 0, st>>>(tokens, token_offsets, block_offsets, num_requests,
                                                                   block_size, salt_term, extra, hashes_out, total_blocks);
    wpp_hash_chain_kernel<<<(unsigned)num_requests, 32, 0, st>>>(block_offsets, hashes_out);
    return cudaGetLastError() == cudaSuccess ? WPP_OK : WPP_ERR_CUDA;
}

extern "C" int wpp_hash_blocks_host(const int32_t* tokens, int64_t n_tokens, int32_t block_size, uint64_t salt,
                                    const uint64_t* extra, uint64_t* hashes_out) {
    if (n_tokens < 0 || block_size < 1) return WPP_ERR_INVALID_ARG;
    const int64_t n = n_tokens / block_size;
    if (n == 0) return WPP_OK;
    if (!tokens || !hashes_out) return WPP_ERR_INVALID_ARG;
    uint64_t h = 0;
    for (int64_t b = 0; b < n; ++b) {
        uint64_t d = 0;
        for (int k = 0; k < block_size; ++k) d += token_term(tokens[b * block_size + k], (uint32_t)k);
        h = chain_step(h, d, extra ? extra[b] : 0ull, salt * 0x9E3779B97F4A7C15ull);
        hashes_out[b] = h;
    }
    return WPP_OK;
}

extern "C" int wpp_hint_index_create(wpp_hint_index** out) {
    if (!out) return WPP_ERR_INVALID_ARG;
    *out = new (std::nothrow) wpp_hint_index();
    return *out ? WPP_OK : WPP_ERR_INVALID_ARG;
}
extern "C" int wpp_hint_index_destroy(wpp_hint_index* idx) {
    delete idx;
    return WPP_OK;
}
extern "C" int wpp_hint_index_add(wpp_hint_index* idx, int32_t window, const uint64_t* hashes, int64_t n) {
    if (!idx || n < 0 || (n > 0 && !hashes)) return WPP_ERR_INVALID_ARG;
    for (int64_t i = 0; i < n; ++i) {
        const int s = wpp_hint_index::shard(hashes[i]);
        std::lock_guard<std::mutex> g(idx->lock[s]);
        idx->map[s][Key{window, hashes[i]}] += 1;
    }
    return WPP_OK;
}
extern "C" int wpp_hint_index_remove(wpp_hint_index* idx, int32_t window, const uint64_t* hashes, int64_t n) {
    if (!idx || n < 0 || (n > 0 && !hashes)) return WPP_ERR_INVALID_ARG;
    for (int64_t i = 0; i < n; ++i) {
        const int s = wpp_hint_index::shard(hashes[i]);
        std::lock_guard<std::mutex> g(idx->lock[s]);
        auto it = idx->map[s].find(Key{window, hashes[i]});
        if (it == idx->map[s].end()) continue;
        if (--it->second <= 0) idx->map[s].erase(it);
    }
    return WPP_OK;
}
extern "C" int64_t wpp_hint_index_size(const wpp_hint_index* idx) {
    if (!idx) return -1;
    int64_t n = 0;
    for (int s = 0; s < kShards; ++s) {
        std::lock_guard<std::mutex> g(idx->lock[s]);
        n += (int64_t)idx->map[s].size();
    }
    return n;
}

extern "C" int wpp_hint_probe(const wpp_hint_index* idx, int32_t window, const uint64_t* hashes, int64_t n_blocks,
                              int64_t* matched_blocks, int32_t* probes_or_null) {
    if (!idx || n_blocks < 0 || !matched_blocks || (n_blocks > 0 && !hashes)) return WPP_ERR_INVALID_ARG;
    int32_t probes = 0;
    int64_t lo = 0, hi = n_blocks + 1;          // depth lo matches (0: nothing known), depth hi misses (or is past the end)
    for (int64_t d = 1; d <= n_blocks; d *= 2) {
        ++probes;
        if (idx->has(window, hashes[d - 1])) {
            lo = d;
        } else {
            hi = d;
            break;
        }
    }
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) / 2;
        ++probes;
        if (idx->has(window, hashes[mid - 1])) lo = mid; else hi = mid;
    }
    *matched_blocks = lo;
    if (probes_or_null) *probes_or_null = probes;
    return WPP_OK;
}

extern "C" int wpp_hint_probe_recurrent(const wpp_hint_index* idx, int32_t window, const uint64_t* hashes,
                                        int64_t limit_blocks, int64_t* matched_blocks, int32_t* probes_or_null) {
    if (!idx || limit_blocks < 0 || !matched_blocks || (limit_blocks > 0 && !hashes)) return WPP_ERR_INVALID_ARG;
    int32_t probes = 0;
    int64_t d = limit_blocks;                   // snapshots are sparse: walk back from the attention-limited endpoint
    for (; d >= 1; --d) {
        ++probes;
        if (idx->has(window, hashes[d - 1])) break;
    }
    *matched_blocks = d;
    if (probes_or_null) *probes_or_null = probes;
    return WPP_OK;
}
