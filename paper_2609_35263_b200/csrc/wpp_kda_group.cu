// Recurrent-state (KDA) layer of a chunk in groups of 16 tokens, the state in registers (Section 3.1 update, Section 3.2
// snapshots).  Per request and head the update
//     S_t = (I - beta_t k_t k_t^T) Diag(alpha_t) S_{t-1} + beta_t k_t v_t^T,     o_t = S_t^T q_t
// over a group of tokens [a, e) that starts from the state S, with the decay products G_t = prod_{a <= r <= t} alpha_r,
// Gt_t = G_t / G_{e-1}, Kt = K o Gt, Kh = K / Gt, Qt = Q o Gt, is
//     A = tril(diag(beta) Kt Kh^T, -1),   T = (I + A)^-1 diag(beta),   M = tril(Qt Kh^T),
//     S' = Diag(G_{e-1}) S,     U = T (V - Kt S'),     O = Qt S' + M U,     S <- S' + Kh^T U.
// (Where the first token's own alpha is too small to divide by, it is applied to the state instead and left out of G.)
//
// The columns of S evolve independently, so a warp that owns 16 or 32 columns carries them through the whole chunk
// without talking to another: S^T lives in its registers as the fp32 accumulator of mma.sync, and because the
// accumulator's layout is that of an A operand, the products X = S^T Kt^T, U^T T^T, U^T M^T and U^T Kh chain from
// registers to registers; only the operands that all columns share (Kt, Qt, Kh, T, M) come from shared memory, where
// producer warps of the same CTA leave them a group ahead.  Nothing crosses HBM but the inputs, the outputs and the
// states.
//
// Why mma.sync beside the tensor cores' asynchronous form (wpp_kda_tc.cu), whose rate is eight times higher: with the
// state in tensor memory a step is a chain of hand-overs between the issuing thread, the tensor pipe and the warps that
// scale, split and store, and its operands need a pass of their own in front (14.5 K clocks of an SM per 64 tokens, 144 KB
// written and read back).  Here a group's chain stays inside a warp: 21 K clocks of an SM per 64 tokens in all, no second
// pass.  8 x 2,048 tokens, 32 heads: 744 -> 669 us; 8 x 64: 58 -> 42 us; 1 x 512: 71 -> 56 us (the choice: kda_chunk_form).
// Whole chains leave the last of few rounds of CTAs partly empty, and a longer chain makes the wave late.  Waves of at least
// as many chains as SMs are therefore cut into pieces of whole blocks (the same bits), dealt out a round of chains after the
// other by tickets that the CTAs take as they start; a piece costs about 6 us besides its tokens, so few of them (kda_pieces).  32
// heads, us, whole (or the two passes, where those were taken instead) | cut: 8 x 2,048 672 | 635 (651 with the piece from the
// CTA's index), 6 x 2,048 610 | 476, 5 x 1,000 297 | 248, 16 x 512..1,024 568 | 490, 8 x 1,024..2,048 537 | 480,
// 5 x 1,500..3,000 545 | 500.  In one kernel with the uncut chains the few more registers spilled
// (64 x 256 tokens, uncut, 697 -> 739), so the cut ones have their own.
// What bounds a group (clocks, 5.3 K before the third terms below): the products 3.4 K of which the MMA pipe is busy 2.6 K,
// U 0.4 K, hand-over and outputs 1.2 K; the producers are idle half the time.  Also tried: four column warps of 32 columns with 216 registers
// (809 us: one warp per scheduler waits), one producer warpgroup (660), a thirteenth warp for T and the copies (711: four
// warps in a quarter of the SM leave 128 registers each).
//
// Precision.  Operands are split into two bf16 terms, x = hi + lo (16 significant bits), a product is three MMAs,
// hi hi + hi lo + lo hi (the dropped lo lo is 2^-17 relative), accumulated in fp32; V - Kt S' and T have three terms and
// their small product six MMAs.  The decay products are relative to the group's end because its last keys, whose share in
// the state has decayed least, then have Kh = K to the bit.  Rms error of the states against 64 bits, over their rms, two
// passes | here, 8 x 2,048 tokens x 32 heads: alpha = sigmoid(4 + 2 n) with n normal 5.09e-6 | 4.35e-6, sigmoid(8 + 2 n)
// 6.73e-6 | 5.27e-6, sigmoid(1 + 2 n) 4.30e-6 | 3.60e-6; with products from the group's start and two terms throughout it was
// 6.33e-6, 7.29e-6 and 5.09e-6 at 645 instead of 676 us.
//
// Groups are the 16-token blocks of absolute sequence positions (so a chunk split at such a position reproduces the
// unsplit result bit for bit), cut wherever the state is needed inside a block (a periodic snapshot) and before every
// token that would push a channel's decay product inside the group below 2^-40.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/wpp.h"
#include "wpp_device.h"
#include "wpp_kda_blocks.cuh"
#include "wpp_ptx.cuh"

namespace wpp {
namespace kdag {

constexpr int kL = 16;                 // tokens per group
constexpr int kD = 128;                // d_k = d_v
constexpr float kMinGamma = 9.094947e-13f;       // 2^-40: smallest decay product a group may contain
constexpr float kSafeGamma = 9.5367432e-7f;      // 2^-20: two halves above it need no closer look
// registers per thread of the 128-column CTAs (eight column warps, eight producer warps, launched with 128 each): the
// column warps keep more operands in flight (8 x 2,048 tokens x 32 heads: 128 / 128 660 us, 144 / 112 656, 152 / 104 640,
// 160 / 96 652)
constexpr int kRegsColumn = 152, kRegsProducer = 104;
static_assert(kRegsColumn + kRegsProducer <= 256, "the launch's registers");

// hi/lo split of two fp32 values into two packed bf16 pairs (element 0 in the low half)
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
    hi = pack_bf16x2(x0, x1);
    const float2 d = __ffma2_rn(make_float2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u)), make_float2(-1.f, -1.f), make_float2(x0, x1));
    lo = pack_bf16x2(d.x, d.y);
}
// three terms: 24 significant bits
__device__ __forceinline__ void split3(float x0, float x1, uint32_t& hi, uint32_t& lo, uint32_t& third) {
    hi = pack_bf16x2(x0, x1);
    const float2 d = __ffma2_rn(make_float2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u)), make_float2(-1.f, -1.f), make_float2(x0, x1));
    lo = pack_bf16x2(d.x, d.y);
    const float2 e = __ffma2_rn(make_float2(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u)), make_float2(-1.f, -1.f), d);
    third = pack_bf16x2(e.x, e.y);
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void mma16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void stsm4t(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};"
                 ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}
__device__ __forceinline__ float2 lds2f(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}
// shared memory by 32-bit address.  No memory clobber: behind one, loads would wait for every store before them; volatile
// statements keep their order among themselves and around the barriers.
__device__ __forceinline__ float lds1f(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds1u(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ float4 lds4f(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts1f(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v)); }
__device__ __forceinline__ void sts1u(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v)); }
__device__ __forceinline__ void sts2f(uint32_t addr, float2 v) { asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y)); }
__device__ __forceinline__ int32_t ld_acquire(const int32_t* p) {
    int32_t v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(int32_t* p, int32_t v) { asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ void named_bar(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// barrier of `threads` threads that also tells whether the predicate holds for any of them
__device__ __forceinline__ bool named_bar_or(int id, int threads, bool pred) {
    uint32_t any;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %3, 0;\n\tbarrier.cta.red.or.pred q, %1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(any) : "r"(id), "r"(threads), "r"((uint32_t)pred) : "memory");
    return any != 0u;
}

// byte offset of 16-byte chunk c (0..15) of row t in a tile of 256-byte rows, swizzled so that eight rows' equal chunks
// lie in different banks
__device__ __forceinline__ uint32_t row_off(int t, int c) { return (uint32_t)(t * 256 + ((c ^ (t & 7)) << 4)); }
// byte offset of the 16-byte half h of row t of a 16 x 16 bf16 matrix, swizzled likewise
__device__ __forceinline__ uint32_t sq_off(int t, int h) { return (uint32_t)(t * 32 + ((h ^ ((t >> 2) & 1)) << 4)); }

struct Maps {
    CUtensorMap q, k, v, alpha;        // (channel, head, row): boxes of 16 rows; alpha as pairs of 16-bit elements
};

// A group as the producers hand it to the column warps.
struct Rec {
    int a, e;            // tokens [a, e) of its 16-token block
    int flags;           // kLast: last group of the block; kPre: the first token's alpha is applied to the state first
    int store_slot;      // state slot to write after the group (periodic snapshot), or -1
};
constexpr int kLast = 1, kPre = 2;

// Shared-memory layout.  One stage = the operands of one group; kVH 64-column halves of V (those the CTA's slice lies in).
template <int kVH>
struct StageT {
    static constexpr int kTile = kL * kD * 2;              // 16 tokens x 128 channels of bf16: 4 KB
    static constexpr int kKtH = 0, kKtL = kTile, kQtH = 2 * kTile, kQtL = 3 * kTile, kKhH = 4 * kTile, kKhL = 5 * kTile;
    static constexpr int kV = 6 * kTile;                   // 64-column halves of 128-byte rows (TMA's swizzle)
    static constexpr int kSq = 16 * 32;                    // a 16 x 16 bf16 matrix
    static constexpr int kTH = kV + kVH * (kTile / 2), kTL = kTH + kSq, kT3 = kTL + kSq, kMH = kT3 + kSq, kML = kMH + kSq;
    static constexpr int kEnd = kML + kSq;                 // fp32 [128]: decay product of the whole group
    static constexpr int kPre = kEnd + kD * 4;             // fp32 [128]: alpha of the first token (if `pre`)
    static constexpr int kRec = kPre + kD * 4;
    static constexpr int kBytes = (kRec + (int)sizeof(Rec) + 1023) / 1024 * 1024;
};
// kP producer warpgroups; each has kStages stages, kRaw raw input slots and scratch of its own
template <int kP, int kVH, int kNC, int kKS>
struct Smem {
    using Stage = StageT<kVH>;
    static constexpr int kStages = 2, kRaw = 2;
    static constexpr int kRawAlpha = 0, kRawK = kL * kD * 4, kRawQ = kRawK + kL * kD * 2, kRawBytes = kRawQ + kL * kD * 2;   // 16 KB
    static constexpr int kAt = 16 * 20 * 4;                // A transposed, fp32
    static constexpr int kScratch = kAt + 2 * kD * 4 + 128 + 64;   // + half products, beta (of alternate blocks), first-bad word
    static constexpr int kOffStage = 0;
    static constexpr int kOffRaw = kP * kStages * Stage::kBytes;
    static constexpr int kOffScratch = kOffRaw + kP * kRaw * kRawBytes;
    static constexpr int kScratchBytes = (kScratch + 127) / 128 * 128;
    static constexpr int kOffOut = kOffScratch + kP * kScratchBytes;         // 1 KB per column warp
    static constexpr int kOffXch = kOffOut + kNC * 1024;                       // partial sums of paired column warps
    static constexpr int kXchBytes = kKS == 1 ? 0 : 3 * 4 * 32 * 8 * 4;       // X [parity][warp][8][lane], O [parity][pair][8][lane]
    static constexpr int kOffBars = kOffXch + kXchBytes;
    static constexpr int kNumBars = kP * (2 * kStages + kRaw);
    static constexpr int kOffMisc = kOffBars + 8 * kNumBars;
    static constexpr int kBytes = kOffMisc + 16 + 1024;
    static_assert(kBytes <= 232448, "more shared memory than a CTA can have");
};

// kSlice value columns per CTA; a column warp owns kMT x 16 of them, or kKS warps share 16 of them and half the channels
// each.  The column warps first, then kP producer warpgroups that take blocks in turn.
__host__ __device__ constexpr int col_warps(int slice, int mt, int ks) { return slice / 16 / mt * ks; }
// kCut: the chains are cut into p.pieces pieces.
template <int kSlice, int kMT, int kKS, int kP, int kMinCtas, bool kCut>
__global__ void __launch_bounds__(32 * col_warps(kSlice, kMT, kKS) + 128 * kP, kMinCtas)
kda_group_kernel(const __grid_constant__ Maps maps, const KdaGroupParams p) {
    constexpr int kNC = col_warps(kSlice, kMT, kKS);
    static_assert(kNC % 4 == 0 && (kKS == 1 || (kKS == 2 && kMT == 1 && kNC == 4)), "whole warpgroups of column warps");
    constexpr int kVH = kSlice == kD ? 2 : 1;
    using SM = Smem<kP, kVH, kNC, kKS>;
    using Stage = StageT<kVH>;
    static_assert(kMinCtas * (SM::kBytes + 1024) <= 233472, "shared memory of an SM");
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
    constexpr int kSlices = kD / kSlice;
    const int H = p.num_heads;
    int head = blockIdx.x / kSlices, slice = blockIdx.x % kSlices, req = blockIdx.y;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(sm + SM::kOffMisc);
    volatile int32_t* ticket = reinterpret_cast<volatile int32_t*>(sm + SM::kOffMisc + 4);
    const uint32_t bars = base + SM::kOffBars;
    auto bFull = [&](int w, int s) { return bars + 8 * (w * (2 * SM::kStages + SM::kRaw) + s); };
    auto bEmpty = [&](int w, int s) { return bFull(w, SM::kStages + s); };
    auto bRaw = [&](int w, int s) { return bFull(w, 2 * SM::kStages + s); };
    auto stage_off = [&](int w, int s) { return SM::kOffStage + (w * SM::kStages + s) * Stage::kBytes; };

    // A wave lasts as long as its longest chain, and only the device knows the lengths: every CTA looks at all of them and
    // comes to the same answer.
    if (p.blk_off) {
        bool longer = false;
        for (int i = tid; i < p.num_requests; i += blockDim.x) longer |= p.row_offsets[i + 1] - p.row_offsets[i] > p.longest;
        const bool first_cta = blockIdx.x == 0 && blockIdx.y == 0;
        if (__syncthreads_or(longer)) {
            if (first_cta) scan_block_offsets<32 * kNC + 128 * kP>(p, reinterpret_cast<int*>(sm));
            return;
        }
        if (first_cta && tid == 0) p.blk_off[0] = -1;
    }

    int piece = 0;
    if constexpr (kCut) {
        // A piece waits for the one before it, so that one has to have started: the CTAs take tickets as they start, all first
        // pieces first, and whatever a ticket waits for is a smaller ticket's.  (CUDA does not say in which order CTAs start.)
        if (tid == 0) *ticket = atomicAdd(p.ticket, 1);
        __syncthreads();
        piece = *ticket / (H * p.num_requests);
        const int chain = *ticket % (H * p.num_requests);
        head = chain % H;
        req = chain / H;
        slice = 0;
    }
    const int64_t row0 = p.row_offsets[req];
    const int C = (int)(p.row_offsets[req + 1] - row0);
    const int P = p.prefix_lens ? p.prefix_lens[req] : 0;
    int first_block = P / kL;
    int n_blocks = C > 0 ? (P + C + kL - 1) / kL - first_block : 0;
    bool resumed = false;
    if constexpr (kCut) {
        // this CTA's piece of the chain.  The pieces of a chain are a whole round of chains apart, and the state goes from one to
        // the next through memory.
        const int begin = (int)((int64_t)n_blocks * piece / p.pieces), end = (int)((int64_t)n_blocks * (piece + 1) / p.pieces);
        if (begin == end && (C > 0 || piece > 0)) return;            // (fewer blocks than pieces; an empty chain is the first CTA's)
        resumed = begin > 0;
        first_block += begin;
        n_blocks = end - begin;
    }

    // slot ids: anything outside [-1, num_slots) is reported and treated as -1
    int slot_in = p.state_in[req], slot_out = p.state_out[req];
    if (slot_in < -1 || slot_in >= p.num_slots || slot_out < -1 || slot_out >= p.num_slots) {
        if (p.status && tid == 0) atomicCAS(p.status, 0, WPP_ERR_BOUNDS);
        if (slot_in < -1 || slot_in >= p.num_slots) slot_in = -1;
        if (slot_out < -1 || slot_out >= p.num_slots) slot_out = -1;
    }
    const size_t head_floats = (size_t)kD * kD;
    if (C == 0) {
        // an empty chunk copies the state
        if (slot_out >= 0 && slot_out != slot_in) {
            float4* dst = reinterpret_cast<float4*>(p.state_pool + ((size_t)slot_out * H + head) * head_floats);
            const float4* src = slot_in >= 0
                ? reinterpret_cast<const float4*>(p.state_pool + ((size_t)slot_in * H + head) * head_floats) : nullptr;
            for (int i = slice * blockDim.x + tid; i < (int)(head_floats / 4); i += kSlices * blockDim.x)
                dst[i] = src ? src[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        return;
    }

    if (tid == 0) {
        for (int w = 0; w < kP; ++w) {
            for (int s = 0; s < SM::kStages; ++s) {
                mbar_init(bFull(w, s), 4 + 1);       // four producer warps, and the request for V
                mbar_init(bEmpty(w, s), kNC);        // the column warps
            }
            for (int s = 0; s < SM::kRaw; ++s) mbar_init(bRaw(w, s), 1);
        }
        *abort_flag = 0u;
        fence_barrier_init();
    }
    __syncthreads();

    if (warp >= kNC) {
        // ================================================================ producers
        if constexpr (kNC == 8) setmaxnreg_dec<kRegsProducer>();
        const int w = (warp - kNC) >> 2;                     // which producer warpgroup: blocks w, w + kP, ...
        const int bar_id = 1 + 2 * w;                      // named barriers: 1 + 2w all four warps, 2 + 2w two of them
        const int ptid = tid & 127, pw = warp & 3;
        const int cp = ptid & 63, half = ptid >> 6;        // channels 2cp, 2cp + 1; tokens 8 half .. 8 half + 7 of a block
        // scratch: A transposed, [s][20] (A[t][s] at s * 20 + t); half products [half][64]; beta of alternate blocks [2][16];
        // the first token that must not stay in the group
        const uint32_t s_at = base + SM::kOffScratch + w * SM::kScratchBytes, s_prod = s_at + SM::kAt, s_betas = s_prod + 2 * kD * 4,
                       s_bad = s_betas + 128;
        const int row_p0 = (int)(row0 - P);                // row of sequence position 0 (may be negative)
        auto row_of = [&](int b) { return row_p0 + (first_block + b) * kL; };
        // Copies are requested by the fourth warp, a lane per copy (a thread spends hundreds of clocks on each), at the end of
        // a group, while the first warp is still forming T.
        auto request_raw = [&](int b, int s) {
            const uint32_t dst = base + SM::kOffRaw + (w * SM::kRaw + s) * SM::kRawBytes;
            if (lane == 0) mbar_arrive_expect_tx(bRaw(w, s), SM::kRawBytes);
            __syncwarp();
            if (lane < 3)
                tma_load_3d(dst + (lane == 0 ? SM::kRawAlpha : lane == 1 ? SM::kRawK : SM::kRawQ),
                            lane == 0 ? &maps.alpha : lane == 1 ? &maps.k : &maps.q, bRaw(w, s), 0, head, row_of(b));
            __syncwarp();
        };
        auto request_v = [&](int b, int s) {               // the block's values, for the column warps
            if (lane == 0) mbar_arrive_expect_tx(bFull(w, s), kVH * (Stage::kTile / 2));
            __syncwarp();
            if (lane < kVH)
                tma_load_3d(base + stage_off(w, s) + Stage::kV + lane * (Stage::kTile / 2), &maps.v, bFull(w, s),
                            (kVH == 2 ? lane : slice * kSlice / 64) * 64, head, row_of(b));
            __syncwarp();
        };
        auto beta_of = [&](int b) -> float {               // lanes 0..15 of the fourth warp
            const int pos = (first_block + b) * kL + lane;
            return (b < n_blocks && pos >= P && pos < P + C) ? p.beta[(int64_t)(row_p0 + pos) * H + head] : 0.f;
        };
        if (pw == 3 && w < n_blocks) {
            for (int s = 0; s < SM::kRaw; ++s)
                if (w + s * kP < n_blocks) request_raw(w + s * kP, s);
            request_v(w, 0);
        }
        float beta_next = (pw == 3 && lane < kL) ? beta_of(w) : 0.f;
        constexpr int kAhead = kMinCtas == 2 ? 4 : 8;          // k-steps of the producers' products whose operands are loaded together

        int stage = 0, raw = 0;
        uint32_t ph_stage = 0, ph_raw = 0;
        bool dead = false;
        for (int b = w; b < n_blocks; b += kP) {
            const int t_lo = max(0, P - (first_block + b) * kL), t_hi = min(kL, P + C - (first_block + b) * kL);
            // this thread's channel pair and first token: alpha (fp32), k and q (bf16)
            const uint32_t r_alpha = base + SM::kOffRaw + (w * SM::kRaw + raw) * SM::kRawBytes + SM::kRawAlpha + half * 8 * kD * 4 + cp * 8;
            const uint32_t r_kq = base + SM::kOffRaw + (w * SM::kRaw + raw) * SM::kRawBytes + SM::kRawK + half * 8 * kD * 2 + cp * 4;
            dead |= !mbar_wait(bRaw(w, raw), ph_raw, abort_flag);
            const uint32_t s_beta = s_betas + (b / kP & 1) * kL * 4;       // (the previous block's may still be in use)
            if (pw == 3 && lane < kL) {
                sts1f(s_beta + lane * 4, beta_next);
                beta_next = beta_of(b + kP);
            }
            int a = t_lo;
            while (a < t_hi) {
                // ---- the group [a, e): up to the block's end or the next snapshot position
                int e = t_hi, store_slot = -1;
                bool snap_here = false;
                if (p.snap_interval > 0) {
                    const int pos = (first_block + b) * kL + a;
                    const int64_t next = ((int64_t)(pos / p.snap_interval) + 1) * p.snap_interval;     // tokens folded into S
                    const int64_t d = next - (int64_t)(first_block + b) * kL;
                    if (d <= t_hi) { e = (int)d; snap_here = true; }
                }
                int pre = 0;
                const int e_max = e;
                const uint32_t st = base + stage_off(w, stage);

                // ---- decay products of this thread's two channels and eight tokens, from the group's first token on
                float2 g[8];
                float2 carry, g_end;
                while (true) {
                    float2 acc = make_float2(1.f, 1.f);
                    float least = 1.f;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int t = half * 8 + i;
                        if (t >= a + pre && t < e) {
                            const float2 al = lds2f(r_alpha + i * kD * 4);
                            acc.x *= al.x;
                            acc.y *= al.y;
                        }
                        g[i] = acc;
                        least = fminf(least, fminf(acc.x, acc.y));
                    }
                    sts2f(s_prod + half * kD * 4 + cp * 8, acc);
                    const bool look = named_bar_or(bar_id, 128, !(least >= kSafeGamma) || dead);
                    const float2 p0 = lds2f(s_prod + cp * 8), p1 = lds2f(s_prod + kD * 4 + cp * 8);
                    carry = half ? p0 : make_float2(1.f, 1.f);
                    g_end = make_float2(p0.x * p1.x, p0.y * p1.y);
                    if (!look) break;
                    // ---- rare: some product may have fallen below 2^-40.  The first token where one did ends the group
                    //      before it; if that is the group's own first token, its alpha goes to the state instead.
                    if (ptid == 0) sts1u(s_bad, kL);
                    if (named_bar_or(bar_id, 128, dead)) { dead = true; break; }
                    int bad = kL;
#pragma unroll
                    for (int i = 7; i >= 0; --i) {
                        const int t = half * 8 + i;
                        if (t >= a && t < e && (!(g[i].x * carry.x >= kMinGamma) || !(g[i].y * carry.y >= kMinGamma))) bad = t;
                    }
                    bad = __reduce_min_sync(0xffffffffu, bad);
                    if (lane == 0) asm volatile("red.shared.min.u32 [%0], %1;" ::"r"(s_bad), "r"(bad) : "memory");
                    named_bar(bar_id, 128);
                    bad = (int)lds1u(s_bad);
                    named_bar(bar_id, 128);
                    if (bad >= e) break;
                    if (bad == a) pre = 1; else e = bad;
                }
                if (dead) break;                           // (everybody: the barrier above has told)
                if (e < e_max) snap_here = false;
                if (snap_here && p.snap_slots) {
                    const int n = ((first_block + b) * kL + e) / p.snap_interval - P / p.snap_interval - 1;
                    if (n < p.max_snaps) {
                        const int slot = p.snap_slots[(size_t)req * p.max_snaps + n];
                        if (slot >= 0 && slot < p.num_slots) store_slot = slot;
                        else if (slot != -1 && p.status && ptid == 0) atomicCAS(p.status, 0, WPP_ERR_BOUNDS);
                    }
                }
                if (ptid == 0)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(st + Stage::kRec), "r"(a), "r"(e),
                                 "r"((e == t_hi ? kLast : 0) | (pre ? kPre : 0)), "r"(store_slot));
                // ---- Kt, Qt and Kh as hi/lo bf16 operands; rows outside the group are zero.  (The stores carry no memory
                //      clobber: behind one, every token's loads would wait for the stores of the token before.)
                const uint32_t row_c = st + half * 2048 + cp * 4;
                const float2 r_end = make_float2(rcp_approx(g_end.x), rcp_approx(g_end.y));              // g_end >= 2^-40: finite
                if (half == 0) sts2f(st + Stage::kEnd + cp * 8, g_end);
                if (pre && half == (a >> 3)) sts2f(st + Stage::kPre + cp * 8, lds2f(r_alpha + (a & 7) * kD * 4));
#pragma unroll
                for (int i0 = 0; i0 < 8; i0 += 4) {
                    uint32_t kr[4], qr[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int t = half * 8 + i0 + u;
                        const bool active = t >= a && t < e;
                        kr[u] = active ? lds1u(r_kq + (i0 + u) * kD * 2) : 0u;
                        qr[u] = active ? lds1u(r_kq + SM::kRawQ - SM::kRawK + (i0 + u) * kD * 2) : 0u;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = i0 + u;
                        const float2 k2 = make_float2(__uint_as_float(kr[u] << 16), __uint_as_float(kr[u] & 0xffff0000u));
                        const float2 q2 = make_float2(__uint_as_float(qr[u] << 16), __uint_as_float(qr[u] & 0xffff0000u));
                        const float2 gs = __fmul2_rn(g[i], carry), gt = __fmul2_rn(gs, r_end);
                        const float2 inv = __fmul2_rn(g_end, make_float2(rcp_approx(gs.x), rcp_approx(gs.y)));      // gs >= 2^-40
                        const uint32_t at = (row_c ^ (i << 4)) + i * 256;                        // row_off(8 half + i, cp >> 2)
                        auto put = [&](int at_hi, int at_lo, float2 x) {
                            uint32_t hi, lo;
                            split2(x.x, x.y, hi, lo);
                            asm volatile("st.shared.b32 [%0], %1;" ::"r"(at + at_hi), "r"(hi));
                            asm volatile("st.shared.b32 [%0], %1;" ::"r"(at + at_lo), "r"(lo));
                        };
                        put(Stage::kKtH, Stage::kKtL, __fmul2_rn(k2, gt));
                        put(Stage::kQtH, Stage::kQtL, __fmul2_rn(q2, gt));
                        put(Stage::kKhH, Stage::kKhL, __fmul2_rn(k2, inv));
                    }
                }
                named_bar(bar_id, 128);

                // ---- Kt Kh^T (warps 0, 1) and Qt Kh^T (warps 2, 3), eight columns each
                {
                    const bool is_m = pw >= 2;
                    const int nt = pw & 1;
                    const uint32_t a_hi = st + (is_m ? Stage::kQtH : Stage::kKtH);
                    const int ln7 = lane & 7, l8 = (lane >> 3) & 1, l16 = lane >> 4;
                    const uint32_t row_a = a_hi + (l8 * 8 + ln7) * 256 + ((l16 ^ ln7) << 4);
                    const uint32_t row_b = st + Stage::kKhH + l16 * Stage::kTile + (nt * 8 + ln7) * 256 + ((l8 ^ ln7) << 4);
                    float x0[4] = {0.f, 0.f, 0.f, 0.f}, x1[4] = {0.f, 0.f, 0.f, 0.f}, x2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int k0 = 0; k0 < 8; k0 += kAhead) {
                        uint32_t ah[kAhead][4], al[kAhead][4], bb[kAhead][4];
#pragma unroll
                        for (int u = 0; u < kAhead; ++u) {
                            const int x = ((k0 + u) & 3) << 5, y = ((k0 + u) >> 2) * 128;
                            ldsm4(ah[u], (row_a ^ x) + y);
                            ldsm4(bb[u], (row_b ^ x) + y);
                            ldsm4(al[u], (row_a ^ x) + y + Stage::kTile);
                        }
#pragma unroll
                        for (int u = 0; u < kAhead; ++u) {
                            mma16(x0, ah[u], bb[u][0], bb[u][1]);
                            mma16(x1, ah[u], bb[u][2], bb[u][3]);
                            mma16(x2, al[u], bb[u][0], bb[u][1]);
                        }
                    }
                    const int s = nt * 8 + 2 * (lane & 3);
                    float x[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) x[i] = x0[i] + (x1[i] + x2[i]);
                    if (!is_m) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int t = (lane >> 2) + (i >> 1) * 8, c = s + (i & 1);
                            sts1f(s_at + (c * 20 + t) * 4, (c < t) ? lds1f(s_beta + t * 4) * x[i] : 0.f);         // rows outside [a, e) are zero already
                        }
                        named_bar(bar_id + 1, 64);
                    } else {
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const int t = (lane >> 2) + i * 8;
                            uint32_t hi, lo;
                            split2(s <= t ? x[2 * i] : 0.f, s + 1 <= t ? x[2 * i + 1] : 0.f, hi, lo);
                            const uint32_t off = sq_off(t, nt) + (s & 7) * 2;
                            asm volatile("st.shared.b32 [%0], %1;" ::"r"(st + Stage::kMH + off), "r"(hi));
                            asm volatile("st.shared.b32 [%0], %1;" ::"r"(st + Stage::kML + off), "r"(lo));
                        }
                    }
                }
                // ---- T = (I + A)^-1 diag(beta): columns of the identity pushed through I + A; lane c has rows 0..7 of column c,
                //      lane c + 16 its rows 8..15 (it gets the upper rows' values, as they become final, by shuffles)
                if (pw == 0) {
                    const int c = lane & 15, r0 = (lane >> 4) * 8;
                    float x[8];
#pragma unroll
                    for (int r = 0; r < 8; ++r) x[r] = (r0 + r == c) ? 1.f : 0.f;
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float xq = __shfl_sync(0xffffffffu, x[q], c);
                        const float4 a0 = lds4f(s_at + (q * 20 + r0) * 4), a1 = lds4f(s_at + (q * 20 + r0 + 4) * 4);
                        // (entries at or above the diagonal are zero: rows that are final already do not change)
                        x[0] = fmaf(-a0.x, xq, x[0]); x[1] = fmaf(-a0.y, xq, x[1]);
                        x[2] = fmaf(-a0.z, xq, x[2]); x[3] = fmaf(-a0.w, xq, x[3]);
                        x[4] = fmaf(-a1.x, xq, x[4]); x[5] = fmaf(-a1.y, xq, x[5]);
                        x[6] = fmaf(-a1.z, xq, x[6]); x[7] = fmaf(-a1.w, xq, x[7]);
                    }
#pragma unroll
                    for (int q = 8; q < 15; ++q) {
                        // rows 8..15: the lower half warp's own (the upper one multiplies by zeros it reads itself)
                        const float xq = r0 ? x[q - 8] : 0.f;
                        const float4 a0 = lds4f(s_at + (q * 20 + 8) * 4), a1 = lds4f(s_at + (q * 20 + 12) * 4);
                        x[0] = fmaf(-a0.x, xq, x[0]); x[1] = fmaf(-a0.y, xq, x[1]);
                        x[2] = fmaf(-a0.z, xq, x[2]); x[3] = fmaf(-a0.w, xq, x[3]);
                        x[4] = fmaf(-a1.x, xq, x[4]); x[5] = fmaf(-a1.y, xq, x[5]);
                        x[6] = fmaf(-a1.z, xq, x[6]); x[7] = fmaf(-a1.w, xq, x[7]);
                    }
                    const float bt = (c >= a && c < e) ? lds1f(s_beta + c * 4) : 0.f;
                    const uint32_t dst = st + Stage::kTH + r0 * 32 + (c & 7) * 2;
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        const float v = x[r] * bt;
                        const __nv_bfloat16 hi = __float2bfloat16_rn(v);
                        const float d = v - __bfloat162float(hi);
                        const __nv_bfloat16 lo = __float2bfloat16_rn(d), third = __float2bfloat16_rn(d - __bfloat162float(lo));
                        const uint32_t at = dst + sq_off(r, c >> 3);             // (the swizzle of row r0 + r is that of row r)
                        asm volatile("st.shared.b16 [%0], %1;" ::"r"(at), "h"(__bfloat16_as_ushort(hi)));
                        asm volatile("st.shared.b16 [%0], %1;" ::"r"(at + Stage::kTL - Stage::kTH), "h"(__bfloat16_as_ushort(lo)));
                        asm volatile("st.shared.b16 [%0], %1;" ::"r"(at + Stage::kT3 - Stage::kTH), "h"(__bfloat16_as_ushort(third)));
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bFull(w, stage));
                if (++stage == SM::kStages) { stage = 0; ph_stage ^= 1u; }
                if (pw == 3) {
                    const int next = e < t_hi ? b : b + kP;
                    if (e == t_hi && b + SM::kRaw * kP < n_blocks) request_raw(b + SM::kRaw * kP, raw);    // the raw tile is spent
                    // (the only wait for a free stage: the others learn of it by the barrier behind the decay products)
                    if (next < n_blocks) {
                        if (__all_sync(0xffffffffu, mbar_wait(bEmpty(w, stage), ph_stage ^ 1u, abort_flag))) request_v(next, stage);
                        else dead = true;
                    }
                }
                a = e;
            }
            if (a < t_hi) break;                               // given up: everybody is here
            if (++raw == SM::kRaw) { raw = 0; ph_raw ^= 1u; }
        }
    } else {
        // ================================================================ the state's columns
        if constexpr (kNC == 8) setmaxnreg_inc<kRegsColumn>();
        constexpr int kNT = 16 / kKS;                      // 8-channel tiles per warp
        const int m0 = (kKS == 1 ? warp : (warp >> 1)) * kMT * 16;          // first column inside the slice
        const int kq = kKS == 1 ? 0 : (warp & 1);
        const int col0 = slice * kSlice + m0;              // first column of the state
        const int ch0 = kq * kNT * 8;                      // first channel
        const int gr = lane >> 2, gc = lane & 3;
        // S[m][j]: rows (columns of the state) gr, gr + 8 of m-tile m; channels ch0 + 8j + 2gc, + 1
        float S[kMT][kNT][4];
        {
            const float* src = slot_in >= 0 && !(kCut && resumed) ? p.state_pool + ((size_t)slot_in * H + head) * head_floats + col0 + gr : nullptr;
#pragma unroll
            for (int m = 0; m < kMT; ++m)
#pragma unroll
                for (int j = 0; j < kNT; ++j)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        S[m][j][i] = src ? src[(size_t)(ch0 + 8 * j + 2 * gc + (i & 1)) * kD + m * 16 + (i >> 1) * 8] : 0.f;
        }
        auto store_state = [&](int slot) {
            float* dst = p.state_pool + ((size_t)slot * H + head) * head_floats + col0 + gr;
#pragma unroll
            for (int m = 0; m < kMT; ++m)
#pragma unroll
                for (int j = 0; j < kNT; ++j)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        dst[(size_t)(ch0 + 8 * j + 2 * gc + (i & 1)) * kD + m * 16 + (i >> 1) * 8] = S[m][j][i];
        };
        bool dead = false;
        // The state between pieces, as this warp's threads hold it, and the last block that it has seen.  (Worked out anew at
        // either end: kept across the chain, the addresses cost registers that the groups need.)
        auto between = [&](float4*& hand, int32_t*& seen) {
            const size_t chain = *ticket % (H * p.num_requests);
            hand = p.hand + chain * (head_floats / 4) + warp * (kMT * kNT * 32) + lane;
            seen = p.hand_seen + chain * kNC + warp;
        };
        if (kCut && resumed) {
            float4* hand;
            int32_t* seen;
            between(hand, seen);
            const long long t0 = clock64();
            int32_t at = 0;                  // (negative: the piece before gave up)
            for (uint32_t n = 0; (at = ld_acquire(seen)) != first_block;) {
                if (at < 0 || ((++n & 31u) == 0u && (*abort_flag || clock64() - t0 > WPP_WAIT_LIMIT))) {
                    *abort_flag = 1u;
                    dead = true;
                    break;
                }
            }
            dead = __any_sync(0xffffffffu, dead);
#pragma unroll
            for (int m = 0; m < kMT; ++m)
#pragma unroll
                for (int j = 0; j < kNT; ++j) {
                    const float4 v = __ldcg(hand + (m * kNT + j) * 32);
                    S[m][j][0] = v.x; S[m][j][1] = v.y; S[m][j][2] = v.z; S[m][j][3] = v.w;
                }
        }
        const uint32_t s_out = base + SM::kOffOut + warp * 1024;
        // lane parts of the operand addresses
        const int ln7 = lane & 7, l8 = (lane >> 3) & 1, l16 = lane >> 4;
        int stage[kP];
        uint32_t ph[kP];
#pragma unroll
        for (int w = 0; w < kP; ++w) { stage[w] = 0; ph[w] = 0; }
        uint32_t n_group = 0;
        bool ready = false;
        for (int b = 0; b < n_blocks && !dead; ++b) {
            const int w = b % kP;
            const int64_t row_t0 = row0 + ((int64_t)(first_block + b) * kL - P);
            bool last = false;
            while (!last) {
                int sg = stage[0];
                uint32_t phs = ph[0];
#pragma unroll
                for (int i = 1; i < kP; ++i) if (w == i) { sg = stage[i]; phs = ph[i]; }
                // (the barrier was tested while the group before was being finished: a wait takes hundreds of clocks even when
                // there is nothing to wait for)
                if (!__all_sync(0xffffffffu, ready) && !__all_sync(0xffffffffu, mbar_wait(bFull(w, sg), phs, abort_flag))) {
                    dead = true;
                    if (kKS == 1) break;
                }
                const uint32_t st = base + stage_off(w, sg);
                const int4 rec = *reinterpret_cast<const int4*>(sm + stage_off(w, sg) + Stage::kRec);
                const int a = rec.x, e = rec.y, store_slot = rec.w;
                last = rec.z & kLast;
                if (rec.z & kPre) {
#pragma unroll
                    for (int j = 0; j < kNT; ++j) {
                        const float2 al = lds2f(st + Stage::kPre + (ch0 + 8 * j + 2 * gc) * 4);
#pragma unroll
                        for (int m = 0; m < kMT; ++m) {
                            S[m][j][0] *= al.x; S[m][j][1] *= al.y; S[m][j][2] *= al.x; S[m][j][3] *= al.y;
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < kNT; ++j) {
                    const float2 f = lds2f(st + Stage::kEnd + (ch0 + 8 * j + 2 * gc) * 4);
#pragma unroll
                    for (int m = 0; m < kMT; ++m) {
                        const float2 lo = __fmul2_rn(make_float2(S[m][j][0], S[m][j][1]), f), hi = __fmul2_rn(make_float2(S[m][j][2], S[m][j][3]), f);
                        S[m][j][0] = lo.x; S[m][j][1] = lo.y; S[m][j][2] = hi.x; S[m][j][3] = hi.y;
                    }
                }
                uint32_t th[4], tl[4], t3[4], mh[4], ml[4];
                // lane addresses of the operands of 16 channels 16 k: row_off(.., 2k + ..) is an exclusive or of the low bits
                // (one register per operand family instead of one per k)
                const uint32_t row_a = st + (l16 * 8 + ln7) * 256 + ((l8 ^ ln7) << 4), row_b = st + (l8 * 8 + ln7) * 256 + ((l16 ^ ln7) << 4);
                auto chunk = [&](uint32_t row, int k) { return (row ^ ((k & 3) << 5)) + (k >> 2) * 128 + kq * 128; };
                const uint32_t sq = sq_off(l16 * 8 + ln7, l8);
                // one 16-column tile after the other, everything about it at once: the registers hold one tile's X, O and
                // U beside the state
#pragma unroll
                for (int m = 0; m < kMT; ++m) {
                    // ---- X^T = S^T Kt^T and the first part of O^T, S^T Qt^T
                    float X[2][4], O[2][4];
#pragma unroll
                    for (int n = 0; n < 2; ++n)
#pragma unroll
                        for (int i = 0; i < 4; ++i) X[n][i] = O[n][i] = 0.f;
                    auto split_state = [&](int kt, uint32_t (&ah)[4], uint32_t (&al)[4]) {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            split2(S[m][2 * kt + (i >> 1)][2 * (i & 1)], S[m][2 * kt + (i >> 1)][2 * (i & 1) + 1], ah[i], al[i]);
                    };
                    if constexpr (kKS == 1) {
#pragma unroll
                        for (int kt = 0; kt < kNT / 2; ++kt) {
                            const uint32_t at = chunk(row_a, kt);
                            uint32_t kh[4], kl[4], qh[4], ql[4], ah[4], al[4];
                            ldsm4(kh, at + Stage::kKtH);
                            ldsm4(qh, at + Stage::kQtH);
                            ldsm4(kl, at + Stage::kKtL);
                            ldsm4(ql, at + Stage::kQtL);
                            split_state(kt, ah, al);
                            mma16(X[0], ah, kh[0], kh[1]);
                            mma16(X[1], ah, kh[2], kh[3]);
                            mma16(O[0], ah, qh[0], qh[1]);
                            mma16(O[1], ah, qh[2], qh[3]);
                            mma16(X[0], al, kh[0], kh[1]);
                            mma16(X[1], al, kh[2], kh[3]);
                            mma16(O[0], al, qh[0], qh[1]);
                            mma16(O[1], al, qh[2], qh[3]);
                            mma16(X[0], ah, kl[0], kl[1]);
                            mma16(X[1], ah, kl[2], kl[3]);
                            mma16(O[0], ah, ql[0], ql[1]);
                            mma16(O[1], ah, ql[2], ql[3]);
                        }
                    } else {
                        // The two warps of a column tile add their halves of the channels.  X, which the chain waits for, goes
                        // first (its small terms in accumulators of their own: four chains of MMAs instead of two); O's
                        // products run while the partial sums cross.
                        uint32_t ah[kNT / 2][4], al[kNT / 2][4];
                        float Xl[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
                        uint32_t kh[kNT / 2][4], kl[kNT / 2][4];
#pragma unroll
                        for (int kt = 0; kt < kNT / 2; ++kt) {
                            const uint32_t at = chunk(row_a, kt);
                            ldsm4(kh[kt], at + Stage::kKtH);
                            ldsm4(kl[kt], at + Stage::kKtL);
                        }
#pragma unroll
                        for (int kt = 0; kt < kNT / 2; ++kt) {
                            split_state(kt, ah[kt], al[kt]);
                            mma16(X[0], ah[kt], kh[kt][0], kh[kt][1]);
                            mma16(X[1], ah[kt], kh[kt][2], kh[kt][3]);
                            mma16(Xl[0], ah[kt], kl[kt][0], kl[kt][1]);
                            mma16(Xl[1], ah[kt], kl[kt][2], kl[kt][3]);
                            mma16(Xl[0], al[kt], kh[kt][0], kh[kt][1]);
                            mma16(Xl[1], al[kt], kh[kt][2], kh[kt][3]);
                        }
                        uint32_t qh[kNT / 2][4], ql[kNT / 2][4];
#pragma unroll
                        for (int kt = 0; kt < kNT / 2; ++kt) {
                            const uint32_t at = chunk(row_a, kt);
                            ldsm4(qh[kt], at + Stage::kQtH);
                            ldsm4(ql[kt], at + Stage::kQtL);
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i) X[i >> 2][i & 3] += Xl[i >> 2][i & 3];
                        const int pair = warp >> 1;
                        float4* xch = reinterpret_cast<float4*>(sm + SM::kOffXch) + (n_group & 1) * 256;      // [warp][2][lane]
                        float4* xo = reinterpret_cast<float4*>(sm + SM::kOffXch) + 512 + (n_group & 1) * 128 + pair * 64;
#pragma unroll
                        for (int n = 0; n < 2; ++n) xch[(warp * 2 + n) * 32 + lane] = make_float4(X[n][0], X[n][1], X[n][2], X[n][3]);
                        float Ol[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
                        for (int kt = 0; kt < kNT / 2; ++kt) {
                            mma16(O[0], ah[kt], qh[kt][0], qh[kt][1]);
                            mma16(O[1], ah[kt], qh[kt][2], qh[kt][3]);
                            mma16(Ol[0], ah[kt], ql[kt][0], ql[kt][1]);
                            mma16(Ol[1], ah[kt], ql[kt][2], ql[kt][3]);
                            mma16(Ol[0], al[kt], qh[kt][0], qh[kt][1]);
                            mma16(Ol[1], al[kt], qh[kt][2], qh[kt][3]);
                        }
                        // (named barriers, a tenth of an mbarrier wait; should one warp have given up waiting for the operands, both
                        // learn it here and leave together)
                        if (named_bar_or(1 + 2 * kP + pair, 64, dead)) { dead = true; break; }
                        // (a sum of two terms does not depend on their order: both warps' X have the same bits)
#pragma unroll
                        for (int n = 0; n < 2; ++n) {
                            const float4 o = xch[((warp ^ 1) * 2 + n) * 32 + lane];
                            X[n][0] += o.x; X[n][1] += o.y; X[n][2] += o.z; X[n][3] += o.w;
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i) O[i >> 2][i & 3] += Ol[i >> 2][i & 3];
                        // the first warp's part of O, on its way to the second while both work on U and S
                        if (kq == 0) {
#pragma unroll
                            for (int n = 0; n < 2; ++n) xo[n * 32 + lane] = make_float4(O[n][0], O[n][1], O[n][2], O[n][3]);
                            asm volatile("bar.arrive %0, %1;" ::"r"(3 + 2 * kP + pair), "r"(64) : "memory");
                        }
                    }
                    // ---- U^T = (V - X)^T T^T, O^T += U^T M^T
                    if (m == 0) {
                        ldsm4(th, st + Stage::kTH + sq);
                        ldsm4(tl, st + Stage::kTL + sq);
                        ldsm4(t3, st + Stage::kT3 + sq);
                        ldsm4(mh, st + Stage::kMH + sq);
                        ldsm4(ml, st + Stage::kML + sq);
                    }
                    uint32_t uh[4], ul[4];
                    {
                        const int vc = col0 + m * 16 + l8 * 8;               // 8 columns of V from here, tokens l16 * 8 + ln7
                        uint32_t vv[4], yh[4], yl[4], y3[4];
                        ldsm4t(vv, st + Stage::kV + (kVH == 2 ? vc >> 6 : 0) * (Stage::kTile / 2) + (l16 * 8 + ln7) * 128 + ((((vc & 63) >> 3) ^ ln7) << 4));
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            // register i: tokens (i >> 1) * 8 + 2gc, + 1 of column gr + (i & 1) * 8
                            const int t = (i >> 1) * 8 + 2 * gc;
                            const float y0 = (t >= a && t < e) ? __uint_as_float(vv[i] << 16) - X[i >> 1][(i & 1) * 2] : 0.f;
                            const float y1 = (t + 1 >= a && t + 1 < e) ? __uint_as_float(vv[i] & 0xffff0000u) - X[i >> 1][(i & 1) * 2 + 1] : 0.f;
                            split3(y0, y1, yh[i], yl[i], y3[i]);
                        }
                        float U[2][4], Ul[2][4];
#pragma unroll
                        for (int n = 0; n < 2; ++n) {
                            U[n][0] = U[n][1] = U[n][2] = U[n][3] = 0.f;
                            Ul[n][0] = Ul[n][1] = Ul[n][2] = Ul[n][3] = 0.f;
                            mma16(U[n], yh, th[2 * n], th[2 * n + 1]);
                            mma16(Ul[n], yh, t3[2 * n], t3[2 * n + 1]);
                        }
#pragma unroll
                        for (int n = 0; n < 2; ++n) {
                            mma16(U[n], yl, th[2 * n], th[2 * n + 1]);
                            mma16(Ul[n], yl, tl[2 * n], tl[2 * n + 1]);
                        }
#pragma unroll
                        for (int n = 0; n < 2; ++n) {
                            mma16(Ul[n], y3, th[2 * n], th[2 * n + 1]);
                            mma16(U[n], yh, tl[2 * n], tl[2 * n + 1]);
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            split2(U[i >> 1][2 * (i & 1)] + Ul[i >> 1][2 * (i & 1)], U[i >> 1][2 * (i & 1) + 1] + Ul[i >> 1][2 * (i & 1) + 1], uh[i], ul[i]);
                    }
                    if (kKS == 1 || kq == 1) {
#pragma unroll
                        for (int n = 0; n < 2; ++n) mma16(O[n], uh, mh[2 * n], mh[2 * n + 1]);
#pragma unroll
                        for (int n = 0; n < 2; ++n) mma16(O[n], ul, mh[2 * n], mh[2 * n + 1]);
#pragma unroll
                        for (int n = 0; n < 2; ++n) mma16(O[n], uh, ml[2 * n], ml[2 * n + 1]);
                    }
                    if (m == kMT - 1) {
                        // the next group's stage: of the other producers if this block is done
                        int wn = last ? (w + 1) % kP : w, sn = 0;
                        uint32_t pn = 0;
#pragma unroll
                        for (int i = 0; i < kP; ++i)
                            if (wn == i) { sn = stage[i]; pn = ph[i]; }
                        if (wn == w && ++sn == SM::kStages) { sn = 0; pn ^= 1u; }
                        ready = mbar_test(bFull(wn, sn), pn);
                    }
                    // ---- S <- S' + (U^T Kh)^T
#pragma unroll
                    for (int j2 = 0; j2 < kNT / 2; ++j2) {
                        const uint32_t at = chunk(row_b, j2);
                        uint32_t bh[4], bl[4];
                        ldsm4t(bh, at + Stage::kKhH);
                        ldsm4t(bl, at + Stage::kKhL);
                        mma16(S[m][2 * j2], uh, bh[0], bh[1]);
                        mma16(S[m][2 * j2 + 1], uh, bh[2], bh[3]);
                        mma16(S[m][2 * j2], ul, bh[0], bh[1]);
                        mma16(S[m][2 * j2 + 1], ul, bh[2], bh[3]);
                        mma16(S[m][2 * j2], uh, bl[0], bl[1]);
                        mma16(S[m][2 * j2 + 1], uh, bl[2], bl[3]);
                    }
                    if (m == kMT - 1) {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bEmpty(w, sg));
                    }
                    // ---- the tile's outputs, to be turned round in shared memory
                    if (kKS == 1 || kq == 1) {
                        if constexpr (kKS == 2) {
                            const int pair = warp >> 1;
                            named_bar(3 + 2 * kP + pair, 64);
                            const float4* xo = reinterpret_cast<const float4*>(sm + SM::kOffXch) + 512 + (n_group & 1) * 128 + pair * 64;
#pragma unroll
                            for (int n = 0; n < 2; ++n) {
                                const float4 o = xo[n * 32 + lane];
                                O[n][0] += o.x; O[n][1] += o.y; O[n][2] += o.z; O[n][3] += o.w;
                            }
                        }
                        // matrices: (columns 0-7, tokens 0-7), (8-15, 0-7), (0-7, 8-15), (8-15, 8-15), stored token-major
                        stsm4t(s_out + m * 512 + (l16 * 8 + ln7) * 32 + l8 * 16,
                               pack_bf16x2(O[0][0], O[0][1]), pack_bf16x2(O[0][2], O[0][3]),
                               pack_bf16x2(O[1][0], O[1][1]), pack_bf16x2(O[1][2], O[1][3]));
                    }
                }
                if (dead) break;
                ++n_group;
#pragma unroll
                for (int i = 0; i < kP; ++i)
                    if (w == i && ++stage[i] == SM::kStages) { stage[i] = 0; ph[i] ^= 1u; }
                if (kKS == 1 || kq == 1) {
                    __syncwarp();
#pragma unroll
                    for (int it = 0; it < kMT; ++it) {
                        const int t = it * (32 / (2 * kMT)) + lane / (2 * kMT), c = lane % (2 * kMT);      // 16-byte chunk c of token t
                        const uint4 v = *reinterpret_cast<const uint4*>(sm + SM::kOffOut + warp * 1024 + (c >> 1) * 512 + t * 32 + (c & 1) * 16);
                        if (t >= a && t < e)
                            *reinterpret_cast<uint4*>(p.out + ((row_t0 + t) * H + head) * kD + col0 + c * 8) = v;
                    }
                    __syncwarp();
                }
                if (store_slot >= 0) store_state(store_slot);
            }
        }
        if (kCut && *ticket < (p.pieces - 1) * H * p.num_requests) {
            float4* hand;
            int32_t* seen;
            between(hand, seen);
            if (!dead) {
#pragma unroll
                for (int m = 0; m < kMT; ++m)
#pragma unroll
                    for (int j = 0; j < kNT; ++j) __stcg(hand + (m * kNT + j) * 32, make_float4(S[m][j][0], S[m][j][1], S[m][j][2], S[m][j][3]));
                __threadfence();
                __syncwarp();
            }
            // (a piece that gave up says so: the ones behind it end at once instead of waiting for their own limit one after the other)
            if (lane == 0) st_release(seen, dead ? -1 : first_block + n_blocks);
        } else if (!dead && slot_out >= 0) {
            store_state(slot_out);
        }
    }

    // ---- teardown: every wait above is bounded, so every thread gets here
    __syncthreads();
    if (*abort_flag) {
        const long long t0 = clock64();
        while (clock64() - t0 < 400000) { }     // let copies in flight land
        if (tid == 0 && p.status) atomicCAS(p.status, 0, WPP_ERR_TIMEOUT);
        __syncthreads();
    }
}

template <int kSlice, int kMT, int kKS, int kP, int kMinCtas, bool kCut = false>
static int launch(const Maps& maps, const KdaGroupParams& p, cudaStream_t st) {
    auto kernel = kda_group_kernel<kSlice, kMT, kKS, kP, kMinCtas, kCut>;
    constexpr int kNC = col_warps(kSlice, kMT, kKS), smem = Smem<kP, (kSlice == kD ? 2 : 1), kNC, kKS>::kBytes;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return (int)e;
        attr_set[dev] = true;
    }
    dim3 grid((unsigned)p.num_heads * (kD / kSlice), (unsigned)p.num_requests);
    if (kCut) {
        static_assert(!kCut || (kSlice == kD && kNC == 8), "a CTA per piece; the layout of hand_seen");
        grid = dim3((unsigned)p.num_heads * (unsigned)p.num_requests * (unsigned)p.pieces);
        const size_t words = 1 + (size_t)kNC * p.num_heads * p.num_requests;         // the ticket, then what has been seen
        const cudaError_t e = cudaMemsetAsync(p.ticket, 0, sizeof(int32_t) * words, st);
        if (e != cudaSuccess) return (int)e;
    }
    kernel<<<grid, 32 * kNC + 128 * kP, smem, st>>>(maps, p);
    return (int)cudaGetLastError();
}

}  // namespace kdag
}  // namespace wpp

// maps: q, k, v, alpha with boxes of 16 rows (v: 64 columns, 128-byte swizzle; the others whole rows, no swizzle)
// form 1: CTAs of 128 columns (eight column warps, two producer warpgroups, one CTA per SM): the operands of a group are
//         made once per chain; for waves with enough (request, head) pairs to fill the SMs.
// form 2: 64 columns (four column warps, one producer warpgroup, two CTAs per SM).
// form 3: 32 columns, the channels halved between paired warps: the shortest chain per group, for a few long chains.
extern "C" int wpp_launch_kda_group(const wpp::KdaGroupParams* p, const CUtensorMap* maps, int form, void* stream) {
    using namespace wpp::kdag;
    Maps m;
    m.q = maps[0]; m.k = maps[1]; m.v = maps[2]; m.alpha = maps[3];
    cudaStream_t st = (cudaStream_t)stream;
    if (form == 3) return launch<32, 1, 2, 2, 1>(m, *p, st);
    if (form == 2) return launch<64, 1, 1, 1, 2>(m, *p, st);
    if (p->pieces > 1) return launch<128, 1, 1, 2, 1, true>(m, *p, st);
    return launch<128, 1, 1, 2, 1>(m, *p, st);
}
