// KV append (bit-exact 16-byte vector copies into the reserved pages) and the split-KV combine pass.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "wpp_device.h"
#include "wpp_plan_format.h"
#include "wpp_ptx.cuh"

namespace wpp {

// One thread moves one 16-byte vector of K and the matching vector of V, or kVec of each.  A vector index decomposes as
// (token, kv head, vector within the head row).
// A request whose span on the device (prefix_lens, chunk_lens) is not the span the plan was made for is refused:
// nothing of it is written and the status word becomes WPP_ERR_PLAN_MISMATCH (Section 4.6: a position mismatch
// fails execution instead of writing against the wrong cache state).
//
// What bounds a small append is its chain of dependent loads, a large one HBM.  The new rows, which depend on nothing, are
// asked for first; the request is found by a search whose every step is one load of 32 offsets by the warp (a bisection by
// each thread was up to seven dependent loads), the plan's offsets come with the launch, and a token is divided out once per
// warp.  Append in a graph, us, a bisection in front of the loads | now: 128 x 3 tokens (64/8 heads) 3.4 | 2.7, 32 x 64 4.3 |
// 4.2, 32 x 256 11.8 | 10.4, 32 x 1,024 47.5 | 47.2 (5.7 TB/s).
//
// A grid that the SMs hold at once (`few`: kAppendCtas per SM, which the launch bounds hold the registers to) is set up while the
// kernel before it runs, which is worth 2 us, and lets the attention kernel in as its CTAs end; a larger one starts behind the
// kernel before and lets the attention kernel in once its last CTAs have started (an SM holds half of its eight: 64 registers).
// Pass, us, the latter for all | the former for all: 1 x 128 tokens over 256 (8/2 heads) 14.3 | 12.5, 32 x 64 (64/8) 25.5 |
// 24.6, 5 x 32..276 over 100..4,000 63.3 | 59.7, but 32 x 512 304 | 309.
constexpr int kAppendVec = 4;          // of a large grid (1: 11.2 us for 32 x 256 tokens, 2: 10.5, 8: 13.5)
constexpr int kAppendCtas = 8;         // per SM
template <int kVec>
__global__ void __launch_bounds__(256, kVec == 1 ? kAppendCtas : kAppendCtas / 2) wpp_append_kernel(const AppendParams p) {
    if (!p.few) grid_launch_dependents();
    grid_dependency_wait();
    const char* plan = static_cast<const char*>(p.plan);
    const int32_t* q_offsets = reinterpret_cast<const int32_t*>(plan + p.off_q_offsets);
    const int32_t* plan_prefix = reinterpret_cast<const int32_t*>(plan + p.off_prefix);
    const uint32_t per_token = (uint32_t)(p.num_kv_heads * p.vec_per_row);
    const int64_t total = p.total_new_tokens * per_token;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * kVec;
    for (int64_t first = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u)) * kVec; first < total; first += stride) {
        const int64_t tok0 = first / per_token;                           // of the warp's first vector
        const uint32_t rem0 = (uint32_t)(first - tok0 * per_token);
        int tok[kVec];
        uint32_t h[kVec], c[kVec];
        uint4 kv[kVec], vv[kVec];
#pragma unroll
        for (int u = 0; u < kVec; ++u) {
            const uint32_t r = rem0 + u * 32 + lane, t = r / per_token, in_token = r - t * per_token;
            tok[u] = first + u * 32 + lane < total ? (int)(tok0 + t) : -1;
            h[u] = in_token / (uint32_t)p.vec_per_row;
            c[u] = in_token - h[u] * (uint32_t)p.vec_per_row;
            if (tok[u] < 0) continue;
            const int64_t src = (int64_t)tok[u] * p.kvnew_token_stride + h[u] * p.kvnew_head_stride + c[u];
            kv[u] = p.k_new[src];
            vv[u] = p.v_new[src];
        }
        int lo = 0, hi = p.num_requests;          // largest i with q_offsets[i] <= tok0
        while (hi - lo > 1) {
            const int width = (hi - lo + 31) / 32, i = lo + lane * width;
            const unsigned le = __ballot_sync(0xffffffffu, i < hi && q_offsets[i] <= tok0) | 1u;
            const int last = 31 - __clz((int)le);
            hi = min(hi, lo + (last + 1) * width);
            lo += last * width;
        }
#pragma unroll
        for (int u = 0; u < kVec; ++u) {
            if (tok[u] < 0) continue;
            // a thread's tokens ascend: the next request usually, but empty ones may lie between (strides that double, then halve;
            // a walk over 30,000 of them took 1.8 ms)
            if (lo + 1 < p.num_requests && q_offsets[lo + 1] <= tok[u]) {
                int width = 1;
                for (++lo; lo + width < p.num_requests && q_offsets[lo + width] <= tok[u]; width *= 2) lo += width;
                while ((width /= 2) > 0)
                    if (lo + width < p.num_requests && q_offsets[lo + width] <= tok[u]) lo += width;
            }
            const int P = p.prefix_lens[lo], at = q_offsets[lo];
            if (P != plan_prefix[lo] || p.chunk_lens[lo] != q_offsets[lo + 1] - at) {
                if (p.status) atomicCAS(p.status, 0, WPP_ERR_PLAN_MISMATCH);
                continue;
            }
            const int pos = P + (tok[u] - at);
            const int blk = pos / p.page_size, slot = pos - blk * p.page_size;
            const int page = (blk < p.max_blocks) ? p.block_tables[(int64_t)lo * p.max_blocks + blk] : -1;
            if (page < 0 || page >= p.num_pages) {
                if (p.status) atomicCAS(p.status, 0, WPP_ERR_BOUNDS);
                continue;
            }
            const int64_t dst = page * p.kv_page_stride + h[u] * p.kv_head_stride + slot * p.kv_token_stride + c[u];
            p.k_cache[dst] = kv[u];
            p.v_cache[dst] = vv[u];
        }
    }
}

// Combine: one warp per row of a split half tile, eight rows per block, grid (half tiles, row groups).  Partials are merged
// in increasing split order with weights exp2(lse_s - max lse), so the result does not depend on scheduling.  The pass is
// a read of the partials; what bounds it is how many of them are in flight.  A lane takes the weight of one part (parts
// beyond 32 in further rounds) and then four (head_dim 64: two) columns of every part, eight parts' loads at a time.  One
// block per half tile whose warps walked the rows, a part's scalar loads after the other's, took 23 us for the 272 half
// tiles x 64 rows x 2 parts of 32 x 64 new tokens over 32,768 cached ones.
constexpr int kCombineRows = 8, kCombineBatch = 8;
template <int D>
__global__ void __launch_bounds__(32 * kCombineRows) wpp_combine_kernel(const CombineParams p) {
    constexpr int kV = D / 32;
    grid_dependency_wait();           // (launched while the attention kernel may still be running)
    const char* plan = static_cast<const char*>(p.plan);
    const WppCombine cu = reinterpret_cast<const WppCombine*>(plan + p.off_combine)[blockIdx.x];
    const int lane = threadIdx.x & 31, r = blockIdx.y * kCombineRows + (threadIdx.x >> 5);
    if (r >= cu.rows) return;
    const int64_t tok = (int64_t)reinterpret_cast<const int32_t*>(plan + p.off_q_offsets)[cu.request] + cu.row0 + r;
    const int64_t row = ((int64_t)cu.slot0 * 2 + cu.half) * 128 + cu.lane0 + r;      // + 256 per part
    float m = -INFINITY, wsum = 0.f;
    bool nan = false;                 // some part's scores had one: the row is NaN, as it is when the tile is not cut
    for (int s = lane; s < cu.num_splits; s += 32) {
        const float l = p.ws_lse[row + s * 256];
        nan |= l != l;
        m = fmaxf(m, l);
    }
    nan = __any_sync(0xffffffffu, nan);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float acc[kV];
#pragma unroll
    for (int k = 0; k < kV; ++k) acc[k] = 0.f;
    if (m > -INFINITY) {
        for (int s0 = 0; s0 < cu.num_splits; s0 += 32) {
            const int cnt = min(32, cu.num_splits - s0);
            // a part that saw no key of this row has lse -inf: its O row is not defined and not used (weight -1 here).  One
            // whose weight merely underflows to zero is used: what it holds may be infinite or NaN.
            const float l_mine = lane < cnt ? p.ws_lse[row + (s0 + lane) * 256] : -INFINITY;
            const float w_mine = l_mine == -INFINITY ? -1.f : exp2f(l_mine - m);
            for (int b0 = 0; b0 < cnt; b0 += kCombineBatch) {
                float x[kCombineBatch][kV], w[kCombineBatch];
#pragma unroll
                for (int u = 0; u < kCombineBatch; ++u) {
                    w[u] = __shfl_sync(0xffffffffu, w_mine, (b0 + u) & 31);
                    const bool use = b0 + u < cnt && !(w[u] < 0.f);
                    const float* src = p.ws_o + (row + (int64_t)(s0 + b0 + u) * 256) * D + lane * kV;
                    if constexpr (kV == 4) {
                        const float4 v = use ? *reinterpret_cast<const float4*>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
                        x[u][0] = v.x; x[u][1] = v.y; x[u][2] = v.z; x[u][3] = v.w;
                    } else {
                        const float2 v = use ? *reinterpret_cast<const float2*>(src) : make_float2(0.f, 0.f);
                        x[u][0] = v.x; x[u][1] = v.y;
                    }
                    if (!use) w[u] = 0.f;
                }
#pragma unroll
                for (int u = 0; u < kCombineBatch; ++u) {
                    wsum += w[u];
#pragma unroll
                    for (int k = 0; k < kV; ++k) acc[k] += w[u] * x[u][k];
                }
            }
        }
    }
    const float inv = nan ? NAN : wsum > 0.f ? 1.f / wsum : 0.f;
    __nv_bfloat16* dst = p.out + tok * p.o_token_stride + (int64_t)cu.head * p.o_head_stride + lane * kV;
    if constexpr (kV == 4)
        *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16x2(acc[0] * inv, acc[1] * inv), pack_bf16x2(acc[2] * inv, acc[3] * inv));
    else
        *reinterpret_cast<uint32_t*>(dst) = pack_bf16x2(acc[0] * inv, acc[1] * inv);
    if (p.lse && lane == 0)
        p.lse[tok * p.num_q_heads + cu.head] = wsum > 0.f && !nan ? (m + log2f(wsum)) * 0.6931471805599453f : -INFINITY;
}

// Self-test of the bounded wait every kernel of the library relies on: one warp waits, with a short limit, on
// a barrier that nothing ever arrives on.  The wait must give up, raise the abort flag and let the kernel end
// normally with WPP_ERR_TIMEOUT in the status word - it never hangs and never traps.
__global__ void wpp_selftest_wait_kernel(long long limit_cycles, int32_t* status, long long* waited_cycles) {
    __shared__ uint64_t bar;
    __shared__ uint32_t abort_flag;
    const uint32_t b = smem_u32(&bar);
    if (threadIdx.x == 0) {
        mbar_init(b, 1);
        abort_flag = 0u;
        fence_barrier_init();
    }
    __syncthreads();
    const long long t0 = clock64();
    const bool ok = mbar_wait_limit(b, 0, &abort_flag, limit_cycles);
    const long long t1 = clock64();
    if (!__all_sync(0xffffffffu, ok) && threadIdx.x == 0) {
        if (status) atomicCAS(status, 0, WPP_ERR_TIMEOUT);
        if (waited_cycles) *waited_cycles = t1 - t0;
    }
}

}  // namespace wpp

extern "C" int wpp_launch_selftest_wait(long long limit_cycles, int32_t* status, long long* waited_cycles,
                                        void* stream) {
    wpp::wpp_selftest_wait_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(limit_cycles, status, waited_cycles);
    return (int)cudaGetLastError();
}

extern "C" int wpp_launch_append(const wpp::AppendParams* p, int num_sms, void* stream) {
    const int64_t total = p->total_new_tokens * p->num_kv_heads * p->vec_per_row;
    if (total == 0) return 0;
    wpp::AppendParams q = *p;
    q.few = total <= (int64_t)num_sms * wpp::kAppendCtas * 256;
    const int per_block = q.few ? 256 : 256 * wpp::kAppendVec;
    int64_t blocks = (total + per_block - 1) / per_block;
    const int64_t cap = (int64_t)num_sms * wpp::kAppendCtas;
    if (blocks > cap) blocks = cap;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute overlap;
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &overlap;
    cfg.numAttrs = q.few ? 1 : 0;
    return (int)cudaLaunchKernelEx(&cfg, q.few ? wpp::wpp_append_kernel<1> : wpp::wpp_append_kernel<wpp::kAppendVec>, q);
}

extern "C" int wpp_launch_combine(const wpp::CombineParams* p, int num_combine, void* stream) {
    if (num_combine == 0) return 0;
    const dim3 grid((unsigned)num_combine, (unsigned)((p->max_rows + wpp::kCombineRows - 1) / wpp::kCombineRows));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(32 * wpp::kCombineRows);
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute overlap;
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &overlap;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, p->head_dim == 128 ? wpp::wpp_combine_kernel<128> : wpp::wpp_combine_kernel<64>, *p);
}
