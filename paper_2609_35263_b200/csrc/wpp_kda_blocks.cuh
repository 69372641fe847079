// The 64-token blocks of the recurrent layer's two passes: a request's geometry, and the scan of the requests' block counts.
#pragma once
#include <stdint.h>

namespace wpp {

constexpr int kKdaBlock = 64;

// Geometry of a request's blocks.  Blocks are aligned to absolute sequence positions.
struct ReqBlocks {
    int64_t row0;       // first row of the request in the packed arrays
    int P, C;           // tokens already folded into the resumed state; chunk length
    int first_block;    // P / 64
    int n_blocks;
};
template <class Params>
__device__ __forceinline__ ReqBlocks req_blocks(const Params& p, int req) {
    ReqBlocks g;
    g.row0 = p.row_offsets[req];
    g.C = (int)(p.row_offsets[req + 1] - g.row0);
    g.P = p.prefix_lens ? p.prefix_lens[req] : 0;
    g.first_block = g.P / kKdaBlock;
    g.n_blocks = g.C > 0 ? (g.P + g.C + kKdaBlock - 1) / kKdaBlock - g.first_block : 0;
    return g;
}

// Exclusive scan of the requests' block counts to p.blk_off [R + 1], by one whole CTA; `part`: an int per thread in shared memory.
template <int kThreads, class Params>
__device__ __forceinline__ void scan_block_offsets(const Params& p, int* part) {
    constexpr int n = kThreads;
    const int R = p.num_requests, tid = threadIdx.x;
    const int per = (R + n - 1) / n;
    const int i0 = min(R, tid * per), i1 = min(R, i0 + per);
    int sum = 0;
    for (int i = i0; i < i1; ++i) sum += req_blocks(p, i).n_blocks;
    part[tid] = sum;
    __syncthreads();
    for (int o = 1; o < n; o <<= 1) {
        const int v = tid >= o ? part[tid - o] : 0;
        __syncthreads();
        part[tid] += v;
        __syncthreads();
    }
    int run = part[tid] - sum;
    for (int i = i0; i < i1; ++i) {
        p.blk_off[i] = run;
        run += req_blocks(p, i).n_blocks;
    }
    if (tid == n - 1) p.blk_off[R] = part[n - 1];
}

}  // namespace wpp
