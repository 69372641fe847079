// Chunked-prefill attention for waves of SHORT tiles (few key steps per tile): a second kernel shape.
//
// The main kernel (wpp_attention.cu) owns an SM: 193 KB of shared memory and all of tensor memory per CTA, two
// 128-row halves in flight.  On tiles of one to eight key steps its pipeline never fills: the start of a tile (tile
// hand-out, unit and page-id reads, Q load, first S, first softmax) and its end (epilogue) take longer than the
// steps in between and nothing of the next tile overlaps them.  This kernel turns the trade round: a CTA is small
// - ONE 128-row half, key steps of 64 keys, 99 KB of shared memory, 256 columns of tensor memory, 320 threads - so
// that TWO CTAs share an SM and one CTA's tile start and end hide under the other's steps.  Roles: warps 0-3 and 6-9
// softmax and epilogue (two threads per query row = tensor-memory lane, half of the keys and of O's columns each),
// warp 4 producer (tile hand-out, page gather, TMA), warp 5 issuer of S = Q K^T and O += P V (its first lane).
// S(j+1) is issued as soon as the softmax warps have copied S(j) out, so the exponentials of step j overlap the next
// score product.
//
// What one tile's latency is spent on counts here.  The first item of a CTA is its own (no round trip to a counter), few or
// equally long items are dealt out altogether, which also takes the memset out of the stream, so that the launch and the
// set-up below (barriers, tensor memory) overlap the kernel before (griddepcontrol).  Nothing of the SM is busy for more than
// a third of the time on 32 x 256 tokens (64/8 heads): a warp's own instructions, one after the other, are what an item takes,
// hence two threads per row; and the producer's global reads (unit, lengths, page ids), 1.3 K clocks each, are made an item
// ahead and 32 pages at a time.  Attention call of one wave, us, one thread per row and a read per request | now:
// 1 x 128 over 256 (8/2 heads, d 64) 12.7 | 9.9, 32 x 64 20.7 | 19.2, 32 x 256 106.7 | 96.1.
// Tried: four epilogue warps beside four softmax warps 118 (32 x 256); an issuing warp for each product and two P in turn 106
// (and 9.4 for 1 x 128).
//
// A work item is one half of a planner tile, (unit, half), or the tile if no tile has a second half; the CTAs take items from
// the counter in the workspace in the planner's order.  Arithmetic, masking, lazy rescaling, head packing, split-KV partials and the bounded
// waits are those of the main kernel.
// Tensor memory: S [0, 64)   P [64, 96) (packed bf16)   O [128, 128 + D).
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "wpp_device.h"
#include "wpp_plan_format.h"
#include "wpp_ptx.cuh"

namespace wpp {
namespace small {

// warps 0-3 and 6-9 softmax and epilogue (32 columns of S each: a warp's number mod 4 says which rows), 4 producer, 5 issuer
constexpr int kThreads = 320;
constexpr int kKeys = 64;                 // keys per step
constexpr int kHalfKeys = kKeys / 2;      // ... per softmax thread
constexpr uint32_t kTmemCols = 256;
constexpr uint32_t kColS = 0, kColP = 64, kColO = 128;
constexpr float kRefSlack = 16.f;         // a row keeps its reference while its scores stay below reference + 16 (log2)
constexpr int kRescaleCols = 16;

// What the producer hands to the other roles with an item, derived from its unit and the request's lengths, so that no
// consumer repeats the dependent global reads.  Read as 16-byte words.  A request whose span on the device differs from the
// plan's gets no key steps (see the main kernel).
struct alignas(16) ItemRec {
    int32_t more;                   // 0: no more items
    int32_t n, step0, kv_len;       // 64-key steps, the first one (absolute), keys of the request
    int32_t first_pos, rows;        // last key visible to row 0; rows of a head
    int32_t log_rph, tok0;          // log2 of the tensor rows per head; first token
    int32_t head, prow0;            // first head; first row of the split partials, or -1: the item writes the final output
    int32_t pad[2];
};
template <int D>
struct Cfg {
    static constexpr int kHalves = D / 64;                 // 64-element (128-byte) swizzled column blocks
    static constexpr int kQBytes = 128 * D * 2;            // the 128-row Q tile
    static constexpr int kQHalfBytes = 128 * 128;
    static constexpr int kKVBytes = kKeys * D * 2;         // one K or V step
    static constexpr int kKVHalfBytes = kKeys * 128;
    static constexpr int kSlots = 2;                       // ring slots for K and for V
    static constexpr int kOffK = kQBytes;
    static constexpr int kOffV = kOffK + kSlots * kKVBytes;
    static constexpr int kOffBars = kOffV + kSlots * kKVBytes;
    static constexpr int kTileQ = 3;
    static constexpr int kNumBars = 2 + 4 * kSlots + 9 + 2 * kTileQ;
    static constexpr int kOffRows = (kOffBars + 8 * kNumBars + 15) / 16 * 16;    // float [2][2][128]: what a row's two threads tell each other
    static constexpr int kOffItems = kOffRows + 4 * 128 * 4;
    static constexpr int kOffMisc = kOffItems + (int)sizeof(ItemRec) * kTileQ;
    static constexpr int kUsedBytes = kOffMisc + 16;
    static constexpr int kSmemBytes = kUsedBytes + 1024;   // 99.5 KB at D = 128
};

struct Ring {
    uint32_t stage, phase;
    __device__ __forceinline__ void advance(uint32_t n) {
        if (++stage == n) { stage = 0; phase ^= 1u; }
    }
};

// 32 bytes to global memory, in one piece where the address allows
__device__ __forceinline__ void store32(void* p, const uint32_t (&x)[8], bool wide) {
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     ::"l"(p), "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]) : "memory");
    } else {
        reinterpret_cast<uint4*>(p)[0] = make_uint4(x[0], x[1], x[2], x[3]);
        reinterpret_cast<uint4*>(p)[1] = make_uint4(x[4], x[5], x[6], x[7]);
    }
}
__device__ __forceinline__ int4 lds_int4(uint32_t addr) {
    int4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

template <int D>
__global__ void __launch_bounds__(kThreads, 2)
wpp_attn_small_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_q64,
                      const __grid_constant__ CUtensorMap tm_q32, const __grid_constant__ CUtensorMap tm_q16,
                      const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                      const SmallAttnParams p) {
    using C = Cfg<D>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t sQ = smem_base, sK = smem_base + C::kOffK, sV = smem_base + C::kOffV;
    const uint32_t bars = smem_base + C::kOffBars;
    const uint32_t bQFull = bars, bQEmpty = bars + 8;
    const uint32_t bKFull = bars + 16, bKEmpty = bKFull + 8 * C::kSlots;
    const uint32_t bVFull = bKEmpty + 8 * C::kSlots, bVEmpty = bVFull + 8 * C::kSlots;
    // s_full: S landed; s_free: the 128 rows have copied it out; p_ready: P written (and O rescaled if a reference
    // moved); p_free: O += P V landed (P may be replaced, O may be rescaled); o_final: the item's last product landed;
    // pair: the two warps of 32 rows have left their values for one another
    const uint32_t bSFull = bVEmpty + 8 * C::kSlots, bSFree = bSFull + 8, bPReady = bSFull + 16, bPFree = bSFull + 24,
                   bOFinal = bSFull + 32, bPair = bSFull + 40;
    const uint32_t bTileFull = bSFull + 72, bTileEmpty = bTileFull + 8 * C::kTileQ;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + C::kOffMisc);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    // every role arrives once per warp
    constexpr uint32_t kTileConsumers = 1 + 8;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        mbar_init(bQFull, 1); mbar_init(bQEmpty, 1);
        for (int s = 0; s < C::kSlots; ++s) {
            mbar_init(bKFull + 8 * s, 1); mbar_init(bKEmpty + 8 * s, 1);
            mbar_init(bVFull + 8 * s, 1); mbar_init(bVEmpty + 8 * s, 1);
        }
        mbar_init(bSFull, 1); mbar_init(bSFree, 8); mbar_init(bPReady, 8); mbar_init(bPFree, 1); mbar_init(bOFinal, 1);
        for (int i = 0; i < 4; ++i) mbar_init(bPair + 8 * i, 2);
        for (int i = 0; i < C::kTileQ; ++i) { mbar_init(bTileFull + 8 * i, 1); mbar_init(bTileEmpty + 8 * i, kTileConsumers); }
        *abort_flag = 0u;
        fence_barrier_init();
    }
    if (warp == 5) {
        tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), kTmemCols);
        tmem_relinquish();
    }
    if (warp == 4 && lane == 0) {
        prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v);
        prefetch_tensormap(&tm_q64); prefetch_tensormap(&tm_q32); prefetch_tensormap(&tm_q16);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_launch_dependents();
    grid_dependency_wait();           // (launched while the kernel before may still be running)

    const char* plan = static_cast<const char*>(p.plan);
    const int32_t* q_offsets = reinterpret_cast<const int32_t*>(plan + p.off_q_offsets);
    const int32_t* plan_prefix = reinterpret_cast<const int32_t*>(plan + p.off_prefix);
    const WppUnit* units = reinterpret_cast<const WppUnit*>(plan + p.off_units);
    const int shift = p.item_shift, num_items = p.num_units << shift;
    Ring tile_ring = {0, 0};
    // the next item for a consuming role (a whole warp): its first kWords 16-byte words; false when there is none or the wait
    // was abandoned
    auto next_item = [&](auto& words) -> bool {
        constexpr int kWords = sizeof(words) / sizeof(words[0]);
        const bool ok = mbar_wait(bTileFull + 8 * tile_ring.stage, tile_ring.phase, abort_flag);
        if (!__all_sync(0xffffffffu, ok)) return false;
        const uint32_t rec = smem_base + C::kOffItems + tile_ring.stage * (uint32_t)sizeof(ItemRec);
#pragma unroll
        for (int i = 0; i < kWords; ++i) words[i] = lds_int4(rec + 16 * i);
        __syncwarp();
        if (lane == 0) mbar_arrive(bTileEmpty + 8 * tile_ring.stage);
        tile_ring.advance(C::kTileQ);
        return words[0].x != 0;
    };
    const int B = p.page_size;
    const int log_b = 31 - __clz(B), log_box = min(log_b, 6);        // a K/V box has min(B, 64) rows (as the maps do)

    if (warp == 4) {
        // ================================================================ producer
        // The global reads of an item - unit, then lengths and page ids - are made while the item before is loaded, the
        // page ids 32 at a time (a lane each): an entry read per request was 1.3 K clocks of 2.6 K per key step.
        Ring ring_k = {0, 0}, ring_v = {0, 0};
        uint32_t q_phase = 0;
        bool dead = false;
        int it_next = (int)blockIdx.x, round = 0;           // the first item is this CTA's own; later ids are taken one ahead
        int it = -1, P = 0, C_len = 0, q_off = 0, q_end = 0, plan_P = 0, pid[2] = {0, 0};
        int4 u0, u1, u2;
        u0 = u1 = u2 = make_int4(0, 0, 0, 0);
        auto take_id = [&]() {                              // asks for the id behind it_next
            if (!p.tile_counter) {
                // (rotated from round to round: neighbouring items - the halves of a unit - are not equally long)
                ++round;
                it_next = round * (int)gridDim.x + (int)((blockIdx.x + round) % gridDim.x);
            }
            else if (lane == 0) it_next = (int)(gridDim.x + atomicAdd(p.tile_counter, 1u));
        };
        auto read_unit = [&]() {
            it = __shfl_sync(0xffffffffu, it_next, 0);
            if (it >= num_items) it = -1;
            if (it < 0) return;
            // (units are 8-byte aligned: the header in front of them is 17 times 8 bytes long)
            static_assert(sizeof(WppPlanHeader) % 8 == 0 && sizeof(WppUnit) == 48, "read as 8-byte words");
            const int2* u = reinterpret_cast<const int2*>(units + (it >> shift));
            const int2 a = u[0], b = u[1], c = u[2], d = u[3], e = u[4], f = u[5];
            u0 = make_int4(a.x, a.y, b.x, b.y);             // request, kv_begin, kv_end, split_slot
            u1 = make_int4(c.x, c.y, d.x, d.y);             // row0[2], rows[2]
            u2 = make_int4(e.x, e.y, f.x, f.y);             // head[2], cost, pack
        };
        // page ids of window w of the item: 32 pages from its first one on
        auto read_pages = [&](int w) {
            const int page = ((u0.y * 128) >> log_b) + 32 * w + lane;
            pid[w & 1] = p.block_tables[(int64_t)u0.x * p.max_blocks + min(page, p.max_blocks - 1)];
        };
        auto read_lengths = [&]() {
            if (it < 0) return;
            P = p.prefix_lens[u0.x];
            C_len = p.chunk_lens[u0.x];
            q_off = q_offsets[u0.x];
            q_end = q_offsets[u0.x + 1];
            plan_P = plan_prefix[u0.x];
            read_pages(0);
        };
        read_unit();
        read_lengths();
        while (!dead) {
            int n = 0, step0 = 0, kv_len = 0, row0 = 0, head = 0;
            {
                const bool ok = mbar_wait(bTileEmpty + 8 * tile_ring.stage, tile_ring.phase ^ 1u, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) break;
                ItemRec rec = {};
                if (it >= 0) {
                    const int hf = it & shift, rows = hf ? u1.w : u1.z;
                    row0 = hf ? u1.y : u1.x;
                    head = hf ? u2.y : u2.x;
                    kv_len = P + C_len;
                    step0 = 2 * u0.y;
                    const bool mismatch = P != plan_P || C_len != q_end - q_off;
                    const int end_keys = min(u0.z * 128, P + row0 + rows);               // keys [.., end_keys) can be visible
                    n = rows > 0 && !mismatch ? max(0, (end_keys + kKeys - 1) / kKeys - step0) : 0;
                    if (mismatch && lane == 0 && p.status) atomicCAS(p.status, 0, WPP_ERR_PLAN_MISMATCH);
                    rec.more = 1, rec.n = n, rec.step0 = step0, rec.kv_len = kv_len;
                    rec.first_pos = P + row0, rec.rows = rows, rec.log_rph = 7 - (31 - __clz(u2.w)), rec.tok0 = q_off + row0;
                    rec.head = head, rec.prow0 = rows > 0 && u0.w >= 0 ? (u0.w * 2 + hf) * 128 : -1;
                    take_id();
                }
                if (lane == 0) {
                    *reinterpret_cast<ItemRec*>(smem_gen + C::kOffItems + tile_ring.stage * sizeof(ItemRec)) = rec;
                    mbar_arrive(bTileFull + 8 * tile_ring.stage);
                }
                tile_ring.advance(C::kTileQ);
            }
            if (it < 0) break;
            if (n == 0) {
                read_unit();
                read_lengths();
                continue;
            }
            const int kvh = head / p.group, first_page = (step0 * kKeys) >> log_b, last_page = (kv_len - 1) >> log_b;
            const int log_pack = 31 - __clz(u2.w);
            // one ring slot: the K or the V tile of step j; box b of the step and its column block h go to lane
            // b * kHalves + h
            auto load_tile = [&](const CUtensorMap* tm, int j, Ring& ring, uint32_t s_base, uint32_t full0, uint32_t empty0) -> bool {
                const int key0 = (step0 + j) * kKeys;
                const int keys = min(kKeys, kv_len - key0);                   // keys of the step that exist
                const int cnt = (keys + (1 << log_box) - 1) >> log_box;       // boxes to fetch
                const int bx = lane / C::kHalves, h = lane % C::kHalves;
                const int key_b = key0 + (bx << log_box), page = (key_b >> log_b) - first_page;
                const int even = __shfl_sync(0xffffffffu, pid[0], page & 31), odd = __shfl_sync(0xffffffffu, pid[1], page & 31);
                int id = bx >= cnt ? 0 : page & 32 ? odd : even;
                if (id < 0 || id >= p.num_pages) {
                    if (p.status) atomicCAS(p.status, 0, WPP_ERR_BOUNDS);
                    id = 0;
                }
                const bool ok = mbar_wait(empty0 + 8 * ring.stage, ring.phase ^ 1u, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) return false;
                const uint32_t full = full0 + 8 * ring.stage;
                if (lane == 0) mbar_arrive_expect_tx(full, (uint32_t)(cnt << log_box) * D * 2);
                __syncwarp();
                if (bx < cnt)
                    tma_load_4d(s_base + ring.stage * C::kKVBytes + (bx << log_box) * 128 + h * C::kKVHalfBytes, tm, full,
                                h * 64, key_b & (B - 1), kvh, id);
                ring.advance(C::kSlots);
                return true;
            };
            auto load_q = [&]() -> bool {
                const bool ok = mbar_wait(bQEmpty, q_phase ^ 1u, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) return false;
                q_phase ^= 1u;
                if (lane == 0) mbar_arrive_expect_tx(bQFull, C::kQBytes);
                __syncwarp();
                // head k of the half lands in tensor rows [k*rph, (k+1)*rph): one box of rph rows per head and
                // 64-column block; box b = (head, column block) is issued by lane b (at most 8 x 2)
                const CUtensorMap* qm = log_pack == 0 ? &tm_q : log_pack == 1 ? &tm_q64 : log_pack == 2 ? &tm_q32 : &tm_q16;
                if (lane < (C::kHalves << log_pack)) {
                    const int k = lane / C::kHalves, h = lane % C::kHalves;
                    // (more places than heads in the group: the last head again, into rows that nobody stores)
                    tma_load_3d(sQ + h * C::kQHalfBytes + k * (128 >> log_pack) * 128, qm, bQFull, h * 64, head + min(k, p.group - 1), q_off + row0);
                }
                return true;
            };
            // the queries need no page ids: they go first when their buffer is free already (the usual case after a
            // short item), else the first K tile goes while the previous item still holds the Q buffer
            const bool q_first = __all_sync(0xffffffffu, mbar_test(bQEmpty, q_phase ^ 1u) != 0u);
            if (q_first && !load_q()) { dead = true; break; }
            if (!load_tile(&tm_k, 0, ring_k, sK, bKFull, bKEmpty)) { dead = true; break; }
            if (!q_first && !load_q()) { dead = true; break; }
            __syncwarp();
            int window = 0;                                 // the last one read
            for (int j = 0; j < n && !dead; ++j) {
                // (V is the later one of the two: when it enters a window, the one before is done with)
                const int w = (((step0 + j) * kKeys >> log_b) - first_page) >> 5;
                if (w == window && first_page + 32 * (w + 1) <= last_page) read_pages(++window);
                if (!load_tile(&tm_v, j, ring_v, sV, bVFull, bVEmpty)) dead = true;
                if (!dead && j + 1 < n && !load_tile(&tm_k, j + 1, ring_k, sK, bKFull, bKEmpty)) dead = true;
            }
            if (dead) break;
            read_unit();
            read_lengths();
        }
    } else if (warp == 5) {
        // ================================================================ issuer of S = Q K^T and O += P V (lane 0)
        Ring ring_k = {0, 0}, ring_v = {0, 0};
        uint32_t q_phase = 0, sfree_phase = 0, pready_phase = 0;
        constexpr uint32_t idesc_qk = idesc_bf16(kKeys, 0, 0), idesc_pv = idesc_bf16(D, 0, 1);
        const uint64_t q_desc = smem_desc_sw128(sQ, 16, 1024);
        const uint64_t k_desc0 = smem_desc_sw128(sK, 16, 1024);                      // + stage * (kKVBytes >> 4)
        const uint64_t v_desc0 = smem_desc_sw128(sV, C::kKVHalfBytes, 1024);
        const uint32_t tS = tmem + kColS, tP = tmem + kColP, tO = tmem + kColO;
        bool dead = false;
        auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
            const bool ok = mbar_wait(bar, parity, abort_flag);
            return __all_sync(0xffffffffu, ok);
        };
        auto issue_s = [&]() -> bool {
            if (!wait(bKFull + 8 * ring_k.stage, ring_k.phase)) return false;
            if (!wait(bSFree, sfree_phase ^ 1u)) return false;       // the landing buffer was copied out
            sfree_phase ^= 1u;
            tc_fence_after();
            if (lane == 0) {
                const uint64_t kd = k_desc0 + (uint64_t)(ring_k.stage * (C::kKVBytes >> 4));
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint64_t qoff = (uint64_t)(((kk >> 2) * C::kQHalfBytes + (kk & 3) * 32) >> 4);
                    const uint64_t koff = (uint64_t)(((kk >> 2) * C::kKVHalfBytes + (kk & 3) * 32) >> 4);
                    if (kk == 0) mma_ss_overwrite(tS, q_desc + qoff, kd + koff, idesc_qk);
                    else mma_ss_accumulate(tS, q_desc + qoff, kd + koff, idesc_qk);
                }
                mma_commit(bSFull);
                mma_commit(bKEmpty + 8 * ring_k.stage);
            }
            ring_k.advance(C::kSlots);
            return true;
        };
        while (!dead) {
            int4 rec[1];
            if (!next_item(rec)) break;
            const int n = rec[0].y, step0 = rec[0].z, kv_len = rec[0].w;
            if (n == 0) continue;
            if (!wait(bQFull, q_phase)) break;
            q_phase ^= 1u;
            if (!issue_s()) break;
            for (int j = 0; j < n; ++j) {
                if (j + 1 < n) { if (!issue_s()) { dead = true; break; } }
                else if (lane == 0) mma_commit(bQEmpty);                   // every S of the item has been issued: Q may be replaced
                if (!wait(bVFull + 8 * ring_v.stage, ring_v.phase)) { dead = true; break; }
                const int valid = kv_len - (step0 + j) * kKeys;          // keys of this step that exist
                if (valid < kKeys) {
                    // rows past the end of the sequence may hold anything (stale slots, boxes never fetched): zero
                    // them so that 0 * garbage cannot reach O
                    uint8_t* vg = smem_gen + C::kOffV + ring_v.stage * C::kKVBytes;
                    for (int h = 0; h < C::kHalves; ++h)
                        for (int i = valid * 8 + lane; i < kKeys * 8; i += 32)
                            *reinterpret_cast<uint4*>(vg + h * C::kKVHalfBytes + i * 16) = make_uint4(0, 0, 0, 0);
                    fence_proxy_async_smem();
                }
                if (!wait(bPReady, pready_phase)) { dead = true; break; }                // P written, O fixed
                pready_phase ^= 1u;
                __syncwarp();
                tc_fence_after();
                if (lane == 0) {
                    const uint64_t vd = v_desc0 + (uint64_t)(ring_v.stage * (C::kKVBytes >> 4));
                    if (j > 0) mma_ts_accumulate(tO, tP, vd, idesc_pv); else mma_ts_overwrite(tO, tP, vd, idesc_pv);
#pragma unroll
                    for (int kk = 1; kk < kKeys / 16; ++kk) mma_ts_accumulate(tO, tP + kk * 8, vd + (uint64_t)(kk * 128), idesc_pv);
                    mma_commit(bPFree);
                    if (j + 1 == n) mma_commit(bOFinal);
                    mma_commit(bVEmpty + 8 * ring_v.stage);
                }
                ring_v.advance(C::kSlots);
            }
        }
    } else {
        // ================================================================ softmax and epilogue (two threads per query row)
        const int quarter = warp & 3, half = warp >= 6 ? 1 : 0, r = quarter * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
        float* const rows = reinterpret_cast<float*>(smem_gen + C::kOffRows) + r;
        uint32_t s_phase = 0, pf_phase = 0, of_phase = 0, turn = 0;
        // the value of the row's other thread; two places in turn, so that one wait is enough
        auto exchange = [&](float mine, float& other) -> bool {
            float* const at = rows + turn * 256;
            at[half * 128] = mine;
            __syncwarp();
            if (lane == 0) mbar_arrive(bPair + 8 * quarter);
            const bool ok = mbar_wait(bPair + 8 * quarter, turn, abort_flag);
            turn ^= 1u;
            other = at[(half ^ 1) * 128];
            return __all_sync(0xffffffffu, ok);
        };
        const float c = p.scale_log2;
        const uint64_t c2 = pack2(c, c);
        // rows of the output on 32-byte boundaries: stored a sector at a time
        const bool wide = ((reinterpret_cast<uintptr_t>(p.out) | (uintptr_t)(p.o_token_stride * 2) | (uintptr_t)(p.o_head_stride * 2)) & 31) == 0;
        bool dead = false;
        while (!dead) {
            int4 rec[3];
            if (!next_item(rec)) break;
            const int n = rec[0].y, step0 = rec[0].z, kv_len = rec[0].w, first_pos = rec[1].x;
            const int rr = r & ((1 << rec[1].z) - 1);                    // row inside its head's block
            const int head = rec[2].x + (r >> rec[1].z);
            const bool row_ok = rr < rec[1].y && (r >> rec[1].z) < p.group, split = rec[2].y >= 0;
            const int64_t tok = (int64_t)rec[1].w + rr, prow = (int64_t)rec[2].y + r;
            if (n == 0) {
                // a split part that lies wholly above this half's diagonal (or a refused request): no key is visible
                if (split && row_ok && !half) p.ws_lse[prow] = -INFINITY;
                continue;
            }
            const int row_last = min(first_pos + rr, kv_len - 1);
            float m_ref = -INFINITY, l_run = 0.f, nmc = 0.f;
            for (int j = 0; j < n; ++j) {
                {
                    const bool ok = mbar_wait(bSFull, s_phase, abort_flag);
                    if (!__all_sync(0xffffffffu, ok)) { dead = true; break; }
                }
                s_phase ^= 1u;
                tc_fence_after();
                float s[kHalfKeys];
                tmem_ld32(lane_addr + kColS + half * kHalfKeys, reinterpret_cast<uint32_t*>(s));
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bSFree);
                const int key0 = (step0 + j) * kKeys + half * kHalfKeys;
                if (key0 + kHalfKeys - 1 > first_pos) {       // only steps that touch the diagonal are masked
                    const int limit = row_last - key0;
#pragma unroll
                    for (int i = 0; i < kHalfKeys; ++i) s[i] = (i > limit) ? -INFINITY : s[i];
                }
                float mx[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) mx[k] = fmax3(fmaxf(s[2 * k], s[2 * k + 1]), s[16 + 2 * k], s[17 + 2 * k]);
                float mxx = fmaxf(fmax3(mx[0], mx[1], mx[2]), fmaxf(fmax3(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7])));
                float mx_other;
                if (!exchange(mxx, mx_other)) { dead = true; break; }
                mxx = fmaxf(mxx, mx_other);
                bool waited = false;
                const bool move = (m_ref == -INFINITY) || !(fmaf(mxx, c, nmc) <= kRefSlack);
                if (__any_sync(0xffffffffu, move)) {
                    const float m_new = fmaxf(m_ref, mxx);
                    const float m_safe = (m_new == -INFINITY) ? 0.f : m_new;
                    const float nmc_new = -m_safe * c;
                    const float alpha = (m_ref == -INFINITY) ? 0.f : fast_exp2(nmc_new - nmc);
                    nmc = nmc_new;
                    m_ref = m_new;
                    l_run *= alpha;
                    if (j > 0) {
                        // O may only be touched once the O += P V of step j-1 has landed
                        const bool okp = mbar_wait(bPFree, pf_phase, abort_flag);
                        if (!__all_sync(0xffffffffu, okp)) { dead = true; break; }
                        pf_phase ^= 1u;
                        waited = true;
                        tc_fence_after();
                        if (__any_sync(0xffffffffu, alpha != 1.f)) {
#pragma unroll 1
                            for (int q0 = half * (D / 2); q0 < (half + 1) * (D / 2); q0 += kRescaleCols) {
                                float o[kRescaleCols];
#pragma unroll
                                for (int c8 = 0; c8 < kRescaleCols; c8 += 8)
                                    tmem_ld8(lane_addr + kColO + q0 + c8, reinterpret_cast<uint32_t*>(o) + c8);
                                tmem_wait_ld();
#pragma unroll
                                for (int i = 0; i < kRescaleCols; ++i) o[i] *= alpha;
#pragma unroll
                                for (int c8 = 0; c8 < kRescaleCols; c8 += 8)
                                    tmem_st8(lane_addr + kColO + q0 + c8, reinterpret_cast<uint32_t*>(o) + c8);
                            }
                        }
                    }
                }
                // p = 2^(s*c - m_ref*c) for the thread's keys: bf16 pairs for the tensor cores, fp32 sum
                uint32_t* pk = reinterpret_cast<uint32_t*>(s);
                {
                    const uint64_t nm2 = pack2(nmc, nmc);
                    uint64_t sum2a = pack2(0.f, 0.f), sum2b = pack2(0.f, 0.f);
#pragma unroll
                    for (int i0 = 0; i0 < kHalfKeys / 2; i0 += 8) {
                        uint64_t x2[8];
                        float e[16];
#pragma unroll
                        for (int k = 0; k < 8; ++k) x2[k] = ffma2(pack2(s[2 * (i0 + k)], s[2 * (i0 + k) + 1]), c2, nm2);
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            float x0, x1;
                            unpack2(x2[k], x0, x1);
                            e[2 * k] = fast_exp2(x0);
                            e[2 * k + 1] = fast_exp2(x1);
                        }
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            if (k & 1) sum2b = fadd2(sum2b, pack2(e[2 * k], e[2 * k + 1]));
                            else sum2a = fadd2(sum2a, pack2(e[2 * k], e[2 * k + 1]));
                            pk[i0 + k] = pack_bf16x2(e[2 * k], e[2 * k + 1]);
                        }
                    }
                    float t0, t1;
                    unpack2(fadd2(sum2a, sum2b), t0, t1);
                    l_run += t0 + t1;
                }
                if (!waited && j > 0) {
                    // P(j-1) must have been consumed before P(j) replaces it
                    const bool okp = mbar_wait(bPFree, pf_phase, abort_flag);
                    if (!__all_sync(0xffffffffu, okp)) { dead = true; break; }
                    pf_phase ^= 1u;
                    tc_fence_after();
                }
#pragma unroll
                for (int c8 = 0; c8 < kHalfKeys / 2; c8 += 8) tmem_st8(lane_addr + kColP + half * (kHalfKeys / 2) + c8, pk + c8);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bPReady);
            }
            if (dead) break;
            // ---- epilogue: half of the columns of O each
            float l_other;
            if (!exchange(l_run, l_other)) break;
            l_run = half ? l_other + l_run : l_run + l_other;
            const float inv_l = (l_run > 0.f) ? 1.f / l_run : 0.f;
            const float lse2 = (l_run <= 0.f) ? -INFINITY : (-nmc + log2f(l_run));       // (NaN if one of the row's scores was)
            uint8_t* dst = split ? reinterpret_cast<uint8_t*>(p.ws_o + prow * D + half * (D / 2))
                                 : reinterpret_cast<uint8_t*>(p.out + tok * p.o_token_stride + (int64_t)head * p.o_head_stride + half * (D / 2));
            // the item's last product has landed (which also consumes the last p_free phase)
            {
                bool ok = mbar_wait(bOFinal, of_phase, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) break;
                of_phase ^= 1u;
                ok = mbar_wait(bPFree, pf_phase, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) break;
                pf_phase ^= 1u;
            }
            tc_fence_after();
#pragma unroll 1
            for (int q4 = 0; q4 < D / 64; ++q4) {
                float o[32];
                tmem_ld32(lane_addr + kColO + half * (D / 2) + q4 * 32, reinterpret_cast<uint32_t*>(o));
                tmem_wait_ld();
                if (row_ok && !split) {
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        uint32_t x[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) x[i] = pack_bf16x2(o[16 * w + 2 * i] * inv_l, o[16 * w + 2 * i + 1] * inv_l);
                        store32(dst + q4 * 64 + w * 32, x, wide);
                    }
                } else if (row_ok) {
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        uint32_t x[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) x[i] = __float_as_uint(o[8 * w + i] * inv_l);
                        store32(dst + q4 * 128 + w * 32, x, true);
                    }
                }
                __syncwarp();
            }
            if (row_ok && !half) {
                if (split) p.ws_lse[prow] = lse2;
                else if (p.lse) p.lse[tok * p.num_q_heads + head] = fmaxf(lse2 * 0.6931471805599453f, -INFINITY);
            }
            tc_fence_before();
        }
    }

    // ---- teardown: every loop above is bounded, so every thread gets here
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        const long long t0 = clock64();
        while (clock64() - t0 < 400000) { }     // let copies and tensor-core work in flight land
        if (threadIdx.x == 0 && p.status) atomicCAS(p.status, 0, WPP_ERR_TIMEOUT);
        __syncthreads();
    }
    if (warp == 5) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

template <int D>
static cudaError_t launch(const CUtensorMap* tq, const CUtensorMap& tk, const CUtensorMap& tv, const SmallAttnParams& p,
                          int num_ctas, cudaStream_t stream) {
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(wpp_attn_small_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             Cfg<D>::kSmemBytes);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)num_ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Cfg<D>::kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute overlap;
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &overlap;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, wpp_attn_small_kernel<D>, tq[0], tq[1], tq[2], tq[3], tk, tv, p);
}

}  // namespace small
}  // namespace wpp

// tq: four maps of q with boxes of 128, 64, 32 and 16 rows; tk, tv: maps whose boxes have min(page_size, 64) rows
extern "C" int wpp_launch_attention_small(int head_dim, const CUtensorMap* tq, const CUtensorMap* tk, const CUtensorMap* tv,
                                          const wpp::SmallAttnParams* p, int num_ctas, void* stream) {
    if (head_dim == 128) return (int)wpp::small::launch<128>(tq, *tk, *tv, *p, num_ctas, (cudaStream_t)stream);
    if (head_dim == 64) return (int)wpp::small::launch<64>(tq, *tk, *tv, *p, num_ctas, (cudaStream_t)stream);
    return (int)cudaErrorInvalidValue;
}
