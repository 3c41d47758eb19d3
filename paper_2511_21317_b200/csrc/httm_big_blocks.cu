// Matching and merging for LARGE merging blocks (257 .. 4096 tokens): the paper's own regime of runs of
// n_s = 128 tokens over n_t = 30 frames, 3840 tokens per block (Sec. 3.3, Sec. 4.1).  A block no longer fits one
// warp's stage, and its similarity step (Eq. 1) is a real dense contraction: n tokens x n_dst dst tokens x 64.
//
//   big_scores_kernel   cosine of every src token of a block with every dst token of the block on the 5th-generation
//                       tensor cores (tcgen05.mma, accumulators in tensor memory), fused with the row-wise
//                       arg-max, which weighs the products by the dst tokens' inverse norms: per src token the best dst
//                       and the best cosine (nothing is written for dst tokens and for blocks in which nothing merges)
//   big_select_kernel   the r src tokens with the best cosines merge (Sec. 3.2): exact radix select per block,
//                       ties by position; writes the assignment map
//   big_merge_kernel    mean of every group (Sec. 3.2): tokens sorted by (merged row, position), one warp
//                       gathers the members of a row in that order; writes merged Q / K / V and rank_q
// All three read the reordered copies (a block is a contiguous run of rows there).
#include <cfloat>

#include "httm_internal.h"
#include "httm_launch.cuh"
#include "tc_sm100.cuh"

namespace httm {

namespace {

// ------------------------------------------------------------------------------------------------ shared helpers
__device__ __forceinline__ uint32_t score_key(float s) {   // unsigned keys order like the floats
    const uint32_t b = __float_as_uint(s);
    return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}
// token number (inside its block) of dst d of n_dst dst tokens: the positions j < n_rule with
// floor((j + 1) n_dst / n_rule) > floor(j n_dst / n_rule), i.e. j = ceil((d + 1) n_rule / n_dst) - 1.  n_rule is the
// block length (evenly spaced dst tokens) or n_dst (the first n_dst tokens: first-frame anchoring), see BlockInfo.
__device__ __forceinline__ int dst_position(int d, int n_rule, int nd) { return ((d + 1) * n_rule + nd - 1) / nd - 1; }
__device__ __forceinline__ bool is_dst_position(int j, int n_rule, int nd) {
    return j < n_rule && ((j + 1) * nd) / n_rule > (j * nd) / n_rule;
}

// ------------------------------------------------------------------------------------------------ scores
// cos(i, d) |x_i| = w_d sum_k x_ik x_dk with w_d = 1 / max(|x_d|, 1e-12).  The products of bf16 values are exact in fp32 and add up in
// tensor memory; the arg-max warps multiply by w_d (one rounding).  All dst tokens of a block (at most 1024: 128 KB) stay in shared
// memory, so a token tile is loaded once and its best so far stays in registers.  What bounds it is the arg-max warps' instruction issue and
// latency (a pair of tiles and 128 dst tokens takes an SM about 2500 cycles, 512 of them MMAs: 46 656 such steps on 148 SMs in 407 us at 1.96 GHz), hence:
//  - a warp works on TWO token tiles at a time: the data of a broadcast load of weights goes to every lane, four cycles of the SM's
//    shared-memory port for four columns, and is used twice this way;
//  - two groups of eight warps, each with a score buffer for a pair of tiles and 128 dst tokens (one group: 515 us);
//  - only the src tokens are rows of the contraction (a quarter of the keys are dst tokens), loaded by two warps with cp.async, the first tiles
//    beside the dst tokens;
//  - work items (tensor, head, block) are taken from a counter, the longest first (dealt in rounds one tensor after the other, the longest of
//    148 CTAs had 15 % more than the mean), and an issuing warp for each group (one for both kept them in step: 437 us).
// The four warps of the roles run with 32 registers: nothing they run may be a function of its own, which would not know of that (build.py fails
// where the compiler has made one).
// Measured at 16 heads x 22 blocks of up to 3840 tokens, 384 dst tokens of the queries and 960 of the keys: 611 us with the dst tokens split into three
// scaled planes, 256 at a time, and one group of warps; 467 us with all tokens as rows; 426 us with a function for scores that had been spoilt; 407 us now.
// It spills all the same: ptxas gives the kernel the 96 registers of its launch, and the scores of two tiles with two Best do not fit (234 bytes stored, 360
// loaded per thread; 278 and 404 with PARTS).  The dst tokens chosen are closer to the best in 64 bits
// (1.6 million tokens of three scenes: 26 off the best by up to 4.6e-7 before, 6 by up to 1.2e-7).  Tried and dropped: 64 and 104 registers (456 us),
// no carrying along where no row of the warp improves (491 us at 467).
constexpr int TILE = 128;                        // rows of an operand tile, dst tokens of a chunk
constexpr int TILE_BYTES = TILE * kRowBytes;     // 16 KB
constexpr int SC_GROUPS = 2;                     // groups of arg-max warps (two column halves x four lane quadrants each)
constexpr int SC_THREADS = 128 + SC_GROUPS * 256;   // warps 0 and 1: MMA issuers of the groups, warps 2 and 3: loads of the token tiles and next work item, then the arg-max warps
constexpr int SC_LOADERS = 64;
constexpr int kScoreRoleRegs = 32, kScoreMaxRegs = 112;   // of the 5 x 96 the kernel starts with
constexpr int SC_TMEM_COLS = 512;                // a buffer pair of 2 x 128 columns (by tile of the pair) for each group
constexpr int SC_STAGES = 10;                    // ring of token tiles behind the dst tokens: as many as there is room for, at least five

struct ScoreBars {
    uint64_t a_full[SC_STAGES], a_empty[SC_STAGES];   // ring of token tiles
    uint64_t s_full[SC_GROUPS], s_empty[SC_GROUPS];   // pairs of score buffers
    uint64_t x_full[SC_GROUPS], x_done[SC_GROUPS];    // exchange of the two column halves' results
    uint32_t tmem_base;
    int abort_flag;
};
struct ScoreItem {
    int t;                            // tensor (0: Q, 1: K); -1: no more items
    int n_rule, even;                 // the block's dst rule; evenly spaced
    int nd, n_src;                    // dst and src tokens
    int n_chunks, st0, n_st, n_pairs; // chunks of dst tokens, the item's tiles of src tokens and pairs of them (none where nothing merges in this block)
    int stages, ring;                 // stages of the ring of token tiles and where it begins
    int64_t row0;                     // row of the block's first token in [H][N]
};
constexpr int SC_AREA = kMaxBigDst * kRowBytes + 5 * TILE_BYTES + 8192;    // dst tokens and ring: 960 dst tokens leave six stages
constexpr int SC_OFF_W = SC_AREA;                                // float [dst]: the weights of the dst tokens
constexpr int SC_OFF_XCH = SC_OFF_W + kMaxBigDst * 4;            // [groups][2][128] (best, arg) of column half 1
constexpr int SC_OFF_BARS = SC_OFF_XCH + 2 * 2 * TILE * 8;
constexpr int SC_OFF_ITEMS = SC_OFF_BARS + 384;                  // ScoreItem [2]: this one and the next
constexpr int SC_SMEM = SC_OFF_ITEMS + 2 * 64 + 1024 /*alignment slack*/;
static_assert(sizeof(ScoreBars) <= 384 && sizeof(ScoreItem) <= 64 && kMaxBigDst % TILE == 0 && SC_AREA % 1024 == 0 && SC_SMEM <= 232448, "");

template <bool PARTS>
__device__ __forceinline__ void write_item(ScoreItem* to, const BigMatchArgs& a, int t_first, int item) {
    const int parts = PARTS ? a.parts : 1, per_tensor = a.heads * a.n_blocks * parts;
    if (item >= 2 * per_tensor) {
        to->t = -1;
        return;
    }
    const int t = item < per_tensor ? t_first : 1 - t_first, at = item < per_tensor ? item : item - per_tensor;
    const int rem = at / parts, part = at - rem * parts;
    const BlockInfo bi = a.blocks[a.order[rem / a.heads]];
    const int nd = t == 0 ? bi.nd_q : bi.nd_k, n_src = bi.n - nd;
    const bool merges = (t == 0 ? bi.r_q : bi.r_k) > 0;
    const int tiles = merges ? (n_src + TILE - 1) / TILE : 0, st0 = tiles * part / parts, n_st = tiles * (part + 1) / parts - st0;
    const int ring = (nd + 7) / 8 * 8 * kRowBytes;   // (the last chunk's MMAs read into the ring: masked columns)
    to->t = t;
    to->n_rule = bi.n_rule;
    to->nd = nd;
    to->n_src = n_src;
    to->even = bi.n_rule == bi.n;
    to->n_chunks = n_st > 0 ? (nd + TILE - 1) / TILE : 0;
    to->st0 = st0;
    to->n_st = n_st;
    to->n_pairs = (n_st + 1) / 2;
    to->ring = ring;
    to->stages = min(SC_STAGES, (SC_AREA - ring) / TILE_BYTES);
    to->row0 = (int64_t)(rem % a.heads) * a.n_tokens + bi.start;
}
// x s for two bf16 values packed in a word, s a power of two: exact (but for values that leave the format)
__device__ __forceinline__ uint32_t scale_bf16x2(uint32_t v, float s) {
    const __nv_bfloat162 r = __floats2bfloat162_rn(__uint_as_float(v << 16) * s, __uint_as_float(v & 0xffff0000u) * s);
    return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ bool zero_row(const __nv_bfloat16* x) {
    uint32_t any = 0;
    for (int c = 0; c < 8; ++c) {
        const uint4 v = ld_global(reinterpret_cast<const uint4*>(x) + c);
        any |= v.x | v.y | v.z | v.w;
    }
    return (any & 0x7fff7fffu) == 0;
}
__device__ __forceinline__ void load_async(uint32_t dst, const void* src) {   // 16 bytes
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// floor(x / den), floor((x + step) / den), ..
struct Ramp {
    int value, rest, den, step_value, step_rest;
    __device__ __forceinline__ Ramp(int x, int step, int den_) : den(den_) {
        value = x / den;
        rest = x - value * den;
        step_value = step / den;
        step_rest = step - step_value * den;
    }
    __device__ __forceinline__ void next() {
        value += step_value;
        rest += step_rest;
        if (rest >= den) {
            rest -= den;
            ++value;
        }
    }
};

// A token's best dst so far: its score, the first dst of the group of eight that holds it, and the scores of that group, which tell the
// dst itself once at the end.  The eight scores are carried along by multiplying with zeros and ones on the FMA pipe, which has time:
// looking for the column whenever a row of the warp improves (in nearly every group) takes two cycles of the ALU for each of 75
// selects and compares, and the ALU has the maxima to take.  A score that is not finite would spoil its place among the
// eight for good (0 x inf): in blocks that can have such scores they are brought inside fp32's range first (finite_score).
constexpr int kGroup = 8;
struct Best {
    float score, first_dst;   // (-1: none)
    float2 v[kGroup / 2];
};
__device__ __forceinline__ float finite_score(float s) { return fminf(fmaxf(s, -FLT_MAX), FLT_MAX); }   // -FLT_MAX where s is not a number
__device__ __forceinline__ void take_best(Best& best, float (&s)[32], int first_dst, int valid) {   // dst first_dst + c, c < valid
    if (valid < 32) {   // the block's last dst tokens: -inf for the maxima, zeros for what is carried along
#pragma unroll
        for (int c = 0; c < 32; ++c)
            if (c >= valid) s[c] = -INFINITY;
    }
    float g[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        g[q] = fmaxf(tc::fmax3(tc::fmax3(s[8 * q], s[8 * q + 1], s[8 * q + 2]), s[8 * q + 3], s[8 * q + 4]), tc::fmax3(s[8 * q + 5], s[8 * q + 6], s[8 * q + 7]));
    if (valid < 32) {
#pragma unroll
        for (int c = 0; c < 32; ++c)
            if (c >= valid) s[c] = 0.f;
    }
    const float m = fmaxf(tc::fmax3(g[0], g[1], g[2]), g[3]);
    bool open = m > best.score;   // (ties: lowest dst, the first group that holds the maximum)
    const float keep = open ? 0.f : 1.f;
    float f[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const bool here = open && g[q] == m;
        f[q] = here ? 1.f : 0.f;
        open = open && !here;
    }
    best.score = fmaxf(best.score, m);
    const float base = (float)first_dst;
    best.first_dst = fmaf(best.first_dst, keep, fmaf(f[0], base, f[1] * (base + 8.f)) + fmaf(f[2], base + 16.f, f[3] * (base + 24.f)));
#pragma unroll
    for (int c = 0; c < kGroup / 2; ++c) {
        float2 v = tc::fmul2(best.v[c], make_float2(keep, keep));
#pragma unroll
        for (int q = 0; q < 4; ++q) v = tc::ffma2(make_float2(s[8 * q + 2 * c], s[8 * q + 2 * c + 1]), make_float2(f[q], f[q]), v);
        best.v[c] = v;
    }
}
// PARTS: blocks shared out to several items (launch_big_scores).  Items that begin at a tile of their own cost more spills: in a call with many blocks, 32 976 tokens x 16 heads in
// blocks of up to 1152 tokens, the kernel took 147.5 us, without 145.4.
template <bool PARTS>
__global__ void __launch_bounds__(SC_THREADS, 1)
big_scores_kernel(const BigMatchArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t s_b = tc::smem_addr(smem);   // dst tokens, behind them the ring of token tiles
    float* w_s = reinterpret_cast<float*>(smem + SC_OFF_W);
    float2* xch = reinterpret_cast<float2*>(smem + SC_OFF_XCH);
    ScoreBars* bars = reinterpret_cast<ScoreBars*>(smem + SC_OFF_BARS);
    volatile int* abort_flag = &bars->abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        bars->abort_flag = 0;
        for (int i = 0; i < SC_STAGES; ++i) {
            tc::mbar_init(tc::smem_addr(&bars->a_full[i]), SC_LOADERS);
            tc::mbar_init(tc::smem_addr(&bars->a_empty[i]), 1);
        }
        for (int i = 0; i < SC_GROUPS; ++i) {
            tc::mbar_init(tc::smem_addr(&bars->s_full[i]), 1);
            tc::mbar_init(tc::smem_addr(&bars->s_empty[i]), 256);
            tc::mbar_init(tc::smem_addr(&bars->x_full[i]), 128);
            tc::mbar_init(tc::smem_addr(&bars->x_done[i]), 128);
        }
        tc::fence_barrier_init();
    }
    // Items come in the order of their work, the tensor with more dst tokens first; a CTA takes the next one that nobody has taken.  Warp 2 reads
    // what there is to know about it while the others work on the one before (three dependent loads from memory).
    const int t_first = a.blocks[a.order[0]].nd_k >= a.blocks[a.order[0]].nd_q ? 1 : 0;
    ScoreItem* items = reinterpret_cast<ScoreItem*>(smem + SC_OFF_ITEMS);
    if (warp == 1) tc::tmem_alloc(tc::smem_addr(&bars->tmem_base), SC_TMEM_COLS);
    if (tid == 64) write_item<PARTS>(items, a, t_first, blockIdx.x);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = bars->tmem_base;
    depend_wait();
    dependents_launch();

    // Every role goes through the same items and meets the others twice in each: behind the gather of the dst tokens and at the end.
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kScoreRoleRegs));
        uint32_t fills = 0;                      // parity (bits) of the fills of every ring stage in the items so far
        uint32_t steps_done = 0;                 // issuers: (pair of tiles, chunk) so far, the score buffers' phases
        for (int n_items = 0;; ++n_items) {
            const ScoreItem it = items[n_items & 1];
            if (it.t < 0) break;
            if (warp >= 2) {
                // ---------------------------------------------------------- loads of the src tokens, 128 to a tile, in the image a tiled copy with
                // the 128-byte swizzle would leave; a tile is handed over while the next one's loads are in flight, unless those have to wait for
                // it.  The first tiles are loaded beside the dst tokens.
                const __nv_bfloat16* x = a.xr[it.t] + it.row0 * kHeadDim;
                const int at = tid - 64, c16 = at & 7;
                // src token s is token s + (dst tokens before it): s + floor(s nd / (n - nd)), or s + nd where the first nd tokens are the dst tokens
                const int s0 = PARTS ? it.st0 * TILE : 0;
                Ramp before((s0 + (at >> 3)) * it.nd, SC_LOADERS / 8 * it.nd, max(it.n_src, 1));
                int s = s0 + (at >> 3), handed = 0, hand_st = 0;   // next src token of this thread; tiles handed over, stage of the next
                uint32_t par = fills;
                auto hand_over = [&]() __attribute__((always_inline)) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tensor cores read the rows through the async proxy
                    tc::mbar_arrive(tc::smem_addr(&bars->a_full[hand_st]));
                    ++handed;
                    if (++hand_st == it.stages) hand_st = 0;
                };
                auto load_tile = [&](int st) __attribute__((always_inline)) {
                    if (!__all_sync(0xffffffffu, tc::mbar_wait(tc::smem_addr(&bars->a_empty[st]), (par >> st & 1u) ^ 1u, abort_flag))) return false;
                    par ^= 1u << st;
                    const uint32_t dst = s_b + it.ring + st * TILE_BYTES;
#pragma unroll 4
                    for (int row = at >> 3; row < TILE; row += SC_LOADERS / 8, s += SC_LOADERS / 8, before.next()) {
                        const int pos = s < it.n_src ? s + (it.even ? before.value : it.nd) : 0;   // (behind the last src token: results dropped)
                        load_async(dst + row * kRowBytes + ((c16 ^ (row & 7)) << 4), x + (int64_t)pos * kHeadDim + c16 * 8);
                    }
                    return true;
                };
                const int first = min(it.n_st, 4);
                bool ok = true;
                for (int st = 0; ok && st < first; ++st) ok = load_tile(st);
                if (__syncthreads_or(0)) __syncthreads();
                asm volatile("cp.async.wait_all;" ::: "memory");
                while (ok && handed < first) hand_over();
                if (tid == 64) write_item<PARTS>(items + ((n_items + 1) & 1), a, t_first, (int)gridDim.x + atomicAdd(a.counter, 1));
                __syncwarp();
                for (int i = first, st = first; ok && i < it.n_st; ++i, st = st + 1 < it.stages ? st + 1 : 0) {
                    if (handed < i && !__all_sync(0xffffffffu, tc::mbar_test(tc::smem_addr(&bars->a_empty[st]), (par >> st & 1u) ^ 1u))) {
                        asm volatile("cp.async.wait_all;" ::: "memory");   // (the stage may be waiting for the tile before)
                        hand_over();
                    }
                    if (!(ok = load_tile(st))) break;
                    asm volatile("cp.async.commit_group;" ::: "memory");
                    if (handed < i) {
                        asm volatile("cp.async.wait_group 1;" ::: "memory");
                        hand_over();
                    }
                }
                asm volatile("cp.async.wait_all;" ::: "memory");
                if (ok && handed < it.n_st) hand_over();
            } else {
                // ---------------------------------------------------------- issuer of a group: S = X_tile . D_chunk^T for both tiles of its pairs.
                // (One warp for both groups keeps them in step, and both wait for their scores at the same time.)
                if (__syncthreads_or(0)) __syncthreads();
                if (tc::elect_one()) {
                    constexpr uint32_t idesc = tc::idesc_bf16(128, TILE, false, false);
                    constexpr uint64_t kTileStep = TILE_BYTES >> 4;   // descriptor address fields count 16-byte units
                    const uint64_t da0 = tc::smem_desc_sw128(s_b + it.ring), db0 = tc::smem_desc_sw128(s_b);
                    const int g = warp;
                    const uint32_t t_s = tmem + 2 * g * TILE, full = tc::smem_addr(&bars->s_full[g]), empty = tc::smem_addr(&bars->s_empty[g]);
                    bool ok = true;
                    int st = 2 * g;                                  // ring stage of the pair's first tile (there are at least five)
                    uint32_t par = fills ^ ((1u << st) - 1u);        // parity (bits) of the fills that come next
                    for (int p = g; ok && p < it.n_pairs; p += SC_GROUPS) {
                        const bool two = 2 * p + 1 < it.n_st;
                        const int st0 = st, st1 = st + 1 < it.stages ? st + 1 : 0;
                        ok = tc::mbar_wait(tc::smem_addr(&bars->a_full[st0]), par >> st0 & 1u, abort_flag) &&
                             (!two || tc::mbar_wait(tc::smem_addr(&bars->a_full[st1]), par >> st1 & 1u, abort_flag));
                        const uint64_t da = da0 + (uint64_t)st0 * kTileStep, db = da0 + (uint64_t)st1 * kTileStep;
                        uint64_t dd = db0;
                        for (int chunk = 0; ok && chunk < it.n_chunks; ++chunk, ++steps_done, dd += kTileStep) {
                            if (!(ok = tc::mbar_wait(empty, (steps_done & 1u) ^ 1u, abort_flag))) break;
                            tc::fence_after_sync();
                            tc::mma_ss_c<false>(t_s, da, dd, idesc);   // K = 16 steps over the 64 channels: 32 bytes = 2 descriptor units
                            tc::mma_ss_c<true>(t_s, da + 2, dd + 2, idesc);
                            tc::mma_ss_c<true>(t_s, da + 4, dd + 4, idesc);
                            tc::mma_ss_c<true>(t_s, da + 6, dd + 6, idesc);
                            if (two) {
                                tc::mma_ss_c<false>(t_s + TILE, db, dd, idesc);
                                tc::mma_ss_c<true>(t_s + TILE, db + 2, dd + 2, idesc);
                                tc::mma_ss_c<true>(t_s + TILE, db + 4, dd + 4, idesc);
                                tc::mma_ss_c<true>(t_s + TILE, db + 6, dd + 6, idesc);
                            }
                            tc::mma_commit(full);
                        }
                        if (ok) {
                            tc::mma_commit(tc::smem_addr(&bars->a_empty[st0]));
                            if (two) tc::mma_commit(tc::smem_addr(&bars->a_empty[st1]));
                        }
                        for (int e = 0; e < 2 * SC_GROUPS; ++e) {   // the stages up to this group's next pair
                            par ^= 1u << st;
                            if (++st == it.stages) st = 0;
                        }
                    }
                }
                __syncwarp();
            }
            for (int st = 0; st < it.stages; ++st) fills ^= (uint32_t)((it.n_st - st + it.stages - 1) / it.stages & 1) << st;
            __syncthreads();
            if (*abort_flag) break;   // (the flag is only set between two barriers: same answer in every thread)
        }
    } else {
        // -------------------------------------------------------------- arg-max over the chunk's dst tokens, one thread per token of either tile of a
        // pair and column half
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kScoreMaxRegs));
        const int g = (warp - 4) >> 3, half = ((warp - 4) >> 2) & 1;
        const int row = (warp & 3) * 32 + lane;            // row of the token tile = lane of tensor memory
        const uint32_t t_s = tmem + g * 2 * TILE + half * 64 + ((uint32_t)((warp & 3) * 32) << 16);
        uint32_t steps_done = 0, pairs_done = 0;           // of this group, all items
        for (int n_items = 0;; ++n_items) {
            const ScoreItem& it = items[n_items & 1];
            if (it.t < 0) break;
            const int nd = it.nd, n_src = it.n_src;
            auto src_position = [&](int s) { return s + (it.even ? s * nd / n_src : nd); };   // (see the loads of the tiles)
            const __nv_bfloat16* x = a.xr[it.t] + it.row0 * kHeadDim;
            const float* inv = a.inv_norm[it.t] + it.row0;
            // ---- the dst tokens, in the same image, and their weights
            // (the last chunk's rows behind these belong to the ring of token tiles: columns that are masked)
            const int rows = it.n_chunks > 0 ? nd : 0, at = tid - 128;
            for (int d = at; d < rows; d += SC_THREADS - 128) w_s[d] = ld_global(inv + dst_position(d, it.n_rule, nd));   // (one or two per thread)
            {
                const int c16 = at & 7;
                constexpr int kRowsPerPass = (SC_THREADS - 128) / 8;
                Ramp pos(((at >> 3) + 1) * it.n_rule - 1, kRowsPerPass * it.n_rule, nd);   // dst_position(d) = ceil((d + 1) n_rule / nd) - 1
#pragma unroll 4
                for (int d = at >> 3; d < rows; d += kRowsPerPass, pos.next())
                    load_async(s_b + d * kRowBytes + ((c16 ^ (d & 7)) << 4), x + (int64_t)pos.value * kHeadDim + c16 * 8);
            }
            // Is any norm of the block, of a src or a dst token, outside 2^-39 .. 2^40 and not zero?  (A weight is at most 1e12, just below 2^40, where the
            // token is zero, tiny or not a number; 0: the squared norm overflowed.)  Inside, every product lies in 2^+-80.
            bool far = false;
            const int n_all = rows > 0 ? nd + n_src : 0;
#pragma unroll 4
            for (int j = at; j < n_all; j += SC_THREADS - 128) {
                const float w = ld_global(inv + j);
                far |= w < 0x1p-40f || (w > 0x1p39f && !zero_row(x + (int64_t)j * kHeadDim));
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tensor cores read the rows through the async proxy
            const bool any_far = __syncthreads_or(far);
            if (any_far) {
                // All dst tokens are scaled by a power of two to norms in (1/2, 1], those below the clamp by 2^39: no product with them is beyond the
                // src token's own norm, and none is lost below fp32's range where the weighted one would not be.
                for (int d = at; d < rows; d += SC_THREADS - 128) {
                    const float w = w_s[d];
                    const float scale = __uint_as_float(__float_as_uint(w) & 0x7f800000u);   // 2^floor(log2 w); 0 for w = 0
                    w_s[d] = __uint_as_float((__float_as_uint(w) & 0x007fffffu) | 0x3f800000u);
#pragma unroll 1
                    for (int c = 0; c < 8; ++c) {
                        uint4* piece = reinterpret_cast<uint4*>(smem + d * kRowBytes) + c;
                        const uint4 v = *piece;
                        *piece = make_uint4(scale_bf16x2(v.x, scale), scale_bf16x2(v.y, scale), scale_bf16x2(v.z, scale), scale_bf16x2(v.w, scale));
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncthreads();
            }
            bool ok = true;
            for (int p = g; ok && p < it.n_pairs; p += SC_GROUPS) {
                Best best[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    best[e].score = -INFINITY;
                    best[e].first_dst = -1.f;
#pragma unroll
                    for (int c = 0; c < kGroup / 2; ++c) best[e].v[c] = make_float2(0.f, 0.f);
                }
                for (int chunk = 0; chunk < it.n_chunks; ++chunk, ++steps_done) {
                    ok = __all_sync(0xffffffffu, tc::mbar_wait(tc::smem_addr(&bars->s_full[g]), steps_done & 1u, abort_flag));   // (a warp gives up together)
                    if (!ok) break;
                    tc::fence_after_sync();
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
                        uint32_t raw[2][32];
                        tc::tmem_ld32(t_s + part * 32, raw[0]);
                        tc::tmem_ld32(t_s + TILE + part * 32, raw[1]);   // (behind the block's last tile: old scores, results dropped)
                        tc::tmem_wait_ld();
                        if (part == 1) {
                            tc::fence_before_sync();
                            tc::mbar_arrive(tc::smem_addr(&bars->s_empty[g]));   // the scores are in registers
                        }
                        const int first_dst = chunk * TILE + half * 64 + part * 32;
                        if (first_dst >= nd) continue;                       // (uniform in the warp)
                        const float4* w4 = reinterpret_cast<const float4*>(w_s + first_dst);
                        float s[2][32];
#pragma unroll
                        for (int c = 0; c < 32; c += 4) {
                            const float4 w = w4[c >> 2];
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                const float2 lo = tc::fmul2(make_float2(__uint_as_float(raw[e][c]), __uint_as_float(raw[e][c + 1])), make_float2(w.x, w.y));
                                const float2 hi = tc::fmul2(make_float2(__uint_as_float(raw[e][c + 2]), __uint_as_float(raw[e][c + 3])), make_float2(w.z, w.w));
                                s[e][c] = lo.x;
                                s[e][c + 1] = lo.y;
                                s[e][c + 2] = hi.x;
                                s[e][c + 3] = hi.y;
                            }
                        }
                        if (any_far) {   // (such blocks only: 64 more instructions of the ALU, 7 % of the call at 82 440 tokens if it is all of them)
#pragma unroll
                            for (int e = 0; e < 2; ++e)
#pragma unroll
                                for (int c = 0; c < 32; ++c) s[e][c] = finite_score(s[e][c]);
                        }
                        take_best(best[0], s[0], first_dst, nd - first_dst);
                        take_best(best[1], s[1], first_dst, nd - first_dst);
                    }
                }
                if (!ok) break;
                int arg[2], own[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int s = ((PARTS ? it.st0 : 0) + 2 * p + e) * TILE + row;   // src token
                    own[e] = (!PARTS || 2 * p + e < it.n_st) && s < n_src ? src_position(s) : -1;   // token number inside the block (behind an odd last tile: another item's)
                    int in_group = 0;
#pragma unroll
                    for (int c = kGroup - 1; c >= 0; --c)
                        if ((c & 1 ? best[e].v[c >> 1].y : best[e].v[c >> 1].x) == best[e].score) in_group = c;
                    arg[e] = (int)best[e].first_dst + in_group;
                    if (best[e].score == FLT_MAX) best[e].score = INFINITY;   // (see finite_score)
                    if (best[e].score <= -FLT_MAX) {   // no score is a number
                        best[e].score = -INFINITY;
                        arg[e] = 0;
                    }
                }
                // the two column halves of a token meet: half 1 hands (best, arg) over, half 0 decides (ties: lowest dst)
                const uint32_t turn = pairs_done++ & 1u;
                float2* mine = xch + g * 2 * TILE + row;
                if (half == 1) {
                    ok = __all_sync(0xffffffffu, tc::mbar_wait(tc::smem_addr(&bars->x_done[g]), turn ^ 1u, abort_flag));
                    if (!ok) break;
#pragma unroll
                    for (int e = 0; e < 2; ++e) mine[e * TILE] = make_float2(best[e].score, __int_as_float(arg[e]));
                    tc::mbar_arrive(tc::smem_addr(&bars->x_full[g]));
                } else {
                    ok = __all_sync(0xffffffffu, tc::mbar_wait(tc::smem_addr(&bars->x_full[g]), turn, abort_flag));
                    if (!ok) break;
                    float2 o[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) o[e] = mine[e * TILE];
                    tc::mbar_arrive(tc::smem_addr(&bars->x_done[g]));
                    float own_w[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) own_w[e] = own[e] >= 0 ? ld_global(inv + own[e]) : 0.f;
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float score = best[e].score;
                        const int oarg = __float_as_int(o[e].y);
                        if (o[e].x > score || (o[e].x == score && oarg < arg[e])) {
                            score = o[e].x;
                            arg[e] = oarg;
                        }
                        if (own[e] >= 0) {
                            // (0 where the token's squared norm overflows.  An infinite token's is not a number, whose key orders above all numbers: it
                            // merges first, as in the kernels of smaller blocks.)
                            a.best_key[it.t][it.row0 + own[e]] = score_key(score * own_w[e]);
                            a.best_pos[it.t][it.row0 + own[e]] = dst_position(arg[e], it.n_rule, nd);
                        }
                    }
                }
            }
            __syncthreads();
            if (*abort_flag) break;   // (as above)
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(tmem, SC_TMEM_COLS);
    if (tid == 0 && bars->abort_flag) atomicCAS(a.status, kDevOk, kDevTimeoutBigMatch);
}

// ------------------------------------------------------------------------------------------------ selection
// One CTA per (tensor, head, block); thread i owns tokens 4 i .. 4 i + 3 of the block, so that counts taken in
// thread order are counts in position order.
constexpr int SEL_THREADS = 1024;

// one warp: walking down from the largest of 256 bins, the bin in which the running count reaches `want`
// (1 <= want <= total); *bin_out = that bin, *want_out = want minus the count of all higher bins
__device__ __forceinline__ void pick_bin(const int* h, int want, int* bin_out, int* want_out) {
    const int lane = threadIdx.x & 31, lo = lane * 8;
    int c = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) c += h[lo + i];
    int incl = c;   // this lane's bins and all higher ones
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_down_sync(0xffffffffu, incl, off);
        if (lane + off < 32) incl += o;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, incl >= want);
    if (hit == 0) {   // cannot happen for want <= total; keep the result defined
        if (lane == 0) {
            *bin_out = 0;
            *want_out = 1;
        }
        return;
    }
    if (lane == 31 - __clz(hit)) {
        int above = incl - c, b = lo + 7;
        for (; b > lo; --b) {
            if (above + h[b] >= want) break;
            above += h[b];
        }
        *bin_out = b;
        *want_out = want - above;
    }
}

__global__ void __launch_bounds__(SEL_THREADS, 1) big_select_kernel(const BigMatchArgs a) {
    __shared__ int hist[256];
    __shared__ int warp_sum[32];
    __shared__ int s_bin, s_want;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int per_tensor = a.heads * a.n_blocks;
    const int t = blockIdx.x / per_tensor, h = (blockIdx.x % per_tensor) / a.n_blocks, b = blockIdx.x % a.n_blocks;
    const BlockInfo bi = a.blocks[b];
    const int n = bi.n, r = t == 0 ? bi.r_q : bi.r_k, nd = t == 0 ? bi.nd_q : bi.nd_k;
    const int64_t base = (int64_t)h * a.n_tokens + bi.start;
    depend_wait();
    dependents_launch();
    int32_t* A = a.assign[t] + base;
    if (r == 0) {   // nothing merges: identity
        for (int j = tid; j < n; j += SEL_THREADS) A[j] = bi.start + j;
        return;
    }
    uint32_t key[4];
    bool src[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int j = 4 * tid + e;
        src[e] = j < n && !is_dst_position(j, bi.n_rule, nd);
        key[e] = src[e] ? a.best_key[t][base + j] : 0u;
    }
    const int n_src = n - nd;
    bool merged[4] = {src[0], src[1], src[2], src[3]};
    if (r < n_src) {
        // T = the r-th largest key: radix select, 8 bits a pass
        uint32_t prefix = 0, mask = 0;
        int want = r;
        for (int shift = 24; shift >= 0; shift -= 8) {
            if (tid < 256) hist[tid] = 0;
            __syncthreads();
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool in = src[e] && (key[e] & mask) == prefix;
                const int bin = in ? (int)((key[e] >> shift) & 255u) : -1;
                const unsigned peers = __match_any_sync(0xffffffffu, bin);   // one atomic per distinct bin of the warp
                if (in && lane == __ffs(peers) - 1) atomicAdd(&hist[bin], __popc(peers));
            }
            __syncthreads();
            if (warp == 0) pick_bin(hist, want, &s_bin, &s_want);
            __syncthreads();
            prefix |= (uint32_t)s_bin << shift;
            mask |= 255u << shift;
            want = s_want;
            __syncthreads();   // s_bin, s_want and hist are rewritten in the next pass
        }
        // keys above T merge; of the keys equal to T the first `want` in position order (Sec. 3.2 ties: lowest position)
        int eq = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) eq += (src[e] && key[e] == prefix) ? 1 : 0;
        int incl = eq;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += o;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            int w = warp_sum[lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, w, off);
                if (lane >= off) w += o;
            }
            warp_sum[lane] = w;
        }
        __syncthreads();
        int before = (warp > 0 ? warp_sum[warp - 1] : 0) + incl - eq;   // equal keys at lower positions
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (src[e] && key[e] == prefix) {
                merged[e] = before < want;
                ++before;
            } else {
                merged[e] = src[e] && key[e] > prefix;
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int j = 4 * tid + e;
        if (j < n) {
            int target = j;
            if (merged[e]) {
                target = a.best_pos[t][base + j];
                if (target < 0 || target >= n) {   // cannot happen after the score kernel; never write a bad index
                    atomicCAS(a.status, kDevOk, kDevBadIndex);
                    target = j;
                }
            }
            A[j] = bi.start + target;
        }
    }
}

// ------------------------------------------------------------------------------------------------ merging
// One CTA per (map in {Q, K}, head, block) - the K map also merges V - plus CTAs that copy the special tokens.
// The sorted-group kernels are templated on T, the threads of a CTA, and E, the tokens per thread: a CTA holds one block of up
// to E T tokens, chosen from the largest block of the context: 64 threads for blocks of up to 256 tokens .. 512 for 4096.
// They gather rows from DRAM and are bound by the loads in flight: several CTAs share an SM (1536 threads of at most 40
// registers), so that one gathers while another sorts.
constexpr int kSortedThreads = 1536;   // resident threads per SM the kernels are compiled for (40 registers)
constexpr int kMergeThreads = 1024;    // .. and the merge kernel: at 64 registers nothing of its sums is spilled, and the fewer blocks gather no slower
                                       // (3840-token blocks as below 241 -> 225 us, 64-token ones 36.9 -> 32.8, 128-token ones 71.7 -> 70; the
                                       // deviation kernel, which reads its rows twice and computes more, is better at three CTAs: filter 178 against 195)
__host__ __device__ constexpr int mg_smem_bytes(int N) { return N * 4 /*keys*/ + N * 2 /*row of kept token*/ + (N + 4) * 4 /*segments*/ + 256; }   // N = E T tokens
__host__ __device__ constexpr int of_smem_bytes(int N) { return mg_smem_bytes(N) + N * 2 /*position of every row's kept token*/ + N /*outlier flags*/ + N * 2 /*new representative of every row*/; }

// two channels of a bf16 row
__device__ __forceinline__ float2 unpack2(uint32_t w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// One stable counting pass over the keys of a block by a six-bit digit of their row: warp w holds elements 32 (E w + s) + lane
// (s = 0 .. E - 1), in this order, and hist[digit * (warps + 1) + warp] counts (the odd pitch spreads the digits over the banks).
// Returns every element's place in the sorted order; elements without a key have digit kRadix.
constexpr int kRadix = 64;
template <int T, int E>
__device__ __forceinline__ void radix_places(const int (&digit)[E], int (&place)[E], int* hist, int* warp_tot) {
    constexpr int W = T / 32, PITCH = W + 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll
    for (int i = tid; i < kRadix * PITCH; i += T) hist[i] = 0;
    __syncthreads();
    const unsigned below = (1u << lane) - 1u;
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const unsigned peers = __match_any_sync(0xffffffffu, digit[s]);
        int* h = hist + (digit[s] & (kRadix - 1)) * PITCH + warp;
        const int before = digit[s] < kRadix ? *h : 0;
        place[s] = before + __popc(peers & below);
        __syncwarp();
        if (digit[s] < kRadix && (peers & below) == 0) *h = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // exclusive sum over the counters in (digit, warp) order, two per thread
    const int e0 = 2 * tid, d0 = e0 / W, d1 = (e0 + 1) / W;
    int* h0 = hist + d0 * PITCH + (e0 - d0 * W);
    int* h1 = hist + d1 * PITCH + (e0 + 1 - d1 * W);
    const int c0 = *h0, c1 = *h1;
    int incl = c0 + c1;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += o;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    int base = 0;   // totals of the warps before this one
    {
        const int w = lane < W ? warp_tot[lane] : 0;
        int v = lane < warp ? w : 0;
        base = __reduce_add_sync(0xffffffffu, v);
    }
    const int excl = base + incl - c0 - c1;
    *h0 = excl;
    *h1 = excl + c0;
    __syncthreads();
#pragma unroll
    for (int s = 0; s < E; ++s) place[s] += digit[s] < kRadix ? hist[digit[s] * PITCH + warp] : 0;
}

// The groups of one block from its map A (every thread of the T-thread CTA calls this): merged row of every kept token =
// its rank among the kept tokens in position order (row_of; -1 for merged tokens); all tokens sorted by (merged row,
// position) in keys[] = (row << 12) | position, so that the members of a row are one ascending run; seg[row] = first
// sorted index of the row, seg[n_kept] = n.  rep_of_row (optional) gets the position of every row's kept token; rank_out
// (optional) the merged row of every token plus moff.  Returns the number of kept tokens, at most `limit` (tokens whose
// row would lie beyond it, or whose target is not a kept token, are recorded as a corrupt map and left out).
// The order comes from two stable counting passes over six bits of the row each (one if there are at most 64 rows), so
// it does not depend on scheduling.  A bitonic sort of the keys took 28 us for 3840 tokens (78 rounds with a barrier each).
// At 82 440 tokens x 16 heads in 3840-token blocks, one CTA of 1024 threads per SM: deviation 203 -> 153 us, filter 92 -> 40, merge
// 310 -> 303; with three CTAs of 512 threads per SM, half of which gather while others sort: 144 (now 101), 31 and 212 us.
template <int T, int E>
__device__ int build_groups(const int32_t* A, int block_start, int n, int limit, uint32_t* keys, int16_t* row_of, int* seg, int* warp_sum,
                            int16_t* rep_of_row, int32_t* status, int32_t* rank_out, int moff) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int* hist = seg;   // (the counters lie where the segments go: 64 (T / 32 + 1) <= E T + 4 words)
    int rep[E];
    unsigned kept[E];
    int n_mine = 0;   // kept tokens of this warp
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const int j = (warp * E + s) * 32 + lane;
        rep[s] = -1;
        if (j < n) {
            rep[s] = ld_global(A + j) - block_start;
            if (rep[s] < 0 || rep[s] >= n) {   // corrupt map: record, treat as kept
                atomicCAS(status, kDevOk, kDevBadIndex);
                rep[s] = j;
            }
        }
        kept[s] = __ballot_sync(0xffffffffu, j < n && rep[s] == j);
        n_mine += __popc(kept[s]);
    }
    __syncthreads();   // (the scratch arrays may still be in use by a previous call's readers)
    if (lane == 0) warp_sum[warp] = n_mine;
    __syncthreads();
    const int w = lane < T / 32 ? warp_sum[lane] : 0;
    const int n_kept = min(__reduce_add_sync(0xffffffffu, w), limit);
    int next_row = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0);
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const int j = (warp * E + s) * 32 + lane;
        if (j < n) {
            const bool is_kept = (kept[s] >> lane) & 1u;
            const int row = next_row + __popc(kept[s] & ((1u << lane) - 1u));
            row_of[j] = is_kept ? (int16_t)row : (int16_t)-1;
            if (is_kept && rep_of_row && row < n_kept) rep_of_row[row] = (int16_t)j;
        }
        next_row += __popc(kept[s]);
    }
    __syncthreads();
    uint32_t key[E];
    int digit[E], place[E];
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const int j = (warp * E + s) * 32 + lane;
        key[s] = 0xffffffffu;
        digit[s] = kRadix;
        if (j < n) {
            int row = row_of[rep[s]];
            if (row < 0 || row >= n_kept) {   // target is not a kept token, or more kept tokens than a valid map has
                atomicCAS(status, kDevOk, kDevBadIndex);
                row = n_kept;                 // (at most 4095 then) sorts behind every valid row, is never gathered
            } else if (rank_out) {
                rank_out[j] = moff + row;
            }
            key[s] = ((uint32_t)row << 12) | (uint32_t)j;
            digit[s] = row & (kRadix - 1);
        }
    }
    radix_places<T, E>(digit, place, hist, warp_sum + 32);
#pragma unroll
    for (int s = 0; s < E; ++s)
        if (key[s] != 0xffffffffu) keys[place[s]] = key[s];
    __syncthreads();
    if (n_kept >= kRadix) {   // (uniform; row n_kept may occur)
#pragma unroll
        for (int s = 0; s < E; ++s) {
            const int j = (warp * E + s) * 32 + lane;
            key[s] = j < n ? keys[j] : 0xffffffffu;
            digit[s] = j < n ? (int)(key[s] >> 18) : kRadix;
        }
        radix_places<T, E>(digit, place, hist, warp_sum + 32);   // (its barriers: every key has been read)
#pragma unroll
        for (int s = 0; s < E; ++s)
            if (key[s] != 0xffffffffu) keys[place[s]] = key[s];
        __syncthreads();
    }
    for (int i = tid; i <= n; i += T) {
        const int row = i < n ? (int)(keys[i] >> 12) : n_kept;
        const int prev = i > 0 ? (int)(keys[i - 1] >> 12) : -1;
        if (row != prev && prev < n_kept)   // every row from prev + 1 to row starts here (rows without members cannot occur in a valid map)
            for (int q = prev + 1; q <= min(row, n_kept); ++q) seg[q] = i;
    }
    __syncthreads();
    return n_kept;
}

// Sum of the rows keys[i0 .. i1) (positions in the low 12 bits), eight channels from x on.  Four members are in flight: the gather is
// bound by load latency.  They are added in pairs of pairs, to one of two sums in turn: n / 8 + 4 roundings for n members.  (Added
// one after the other they took n: with one member 2^17 times the others, 2 048 of them left the mean half a step of bf16 off; that
// was a little faster, at 82 440 tokens x 16 heads in 3840-token blocks filter 216 / 221 us, merge 224 / 237 us.)
__device__ __forceinline__ void sum_members(const __nv_bfloat16* x, const uint32_t* keys, int i0, int i1, float2 (&sum)[4]) {
    float2 other[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) sum[e] = other[e] = make_float2(0.f, 0.f);
    auto add_four = [&](int i, float2 (&to)[4]) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[u] = make_uint4(0u, 0u, 0u, 0u);
            if (i + u < i1) v[u] = ld_global(reinterpret_cast<const uint4*>(x + (keys[i + u] & 4095u) * kHeadDim));
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            auto word = [&](int u) { return unpack2(e == 0 ? v[u].x : e == 1 ? v[u].y : e == 2 ? v[u].z : v[u].w); };
            to[e] = tc::fadd2(to[e], tc::fadd2(tc::fadd2(word(0), word(1)), tc::fadd2(word(2), word(3))));
        }
    };
    for (int i = i0; i < i1; i += 8) {
        add_four(i, sum);
        if (i + 4 < i1) add_four(i + 4, other);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) sum[e] = tc::fadd2(sum[e], other[e]);
}

// SHARED: several CTAs for a block (row_shares).  With the distance between a warp's rows known only at run time a call with many blocks, 32 976 tokens x 16 heads in blocks of
// up to 1152 tokens, took 512.2 us, without 510.8.
template <int T, int E, bool SHARED>
__global__ void __launch_bounds__(T, kMergeThreads / T) big_merge_kernel(const MergeArgs a, int sp_chunks, int n_shares) {
    const int shares = SHARED ? n_shares : 1;
    extern __shared__ __align__(16) unsigned char mg_smem[];
    uint32_t* keys = reinterpret_cast<uint32_t*>(mg_smem);                                     // [P] (merged row << 12) | position
    int16_t* row_of = reinterpret_cast<int16_t*>(mg_smem + (E * T) * 4);            // [n] merged row of a kept token, -1
    int* seg = reinterpret_cast<int*>(mg_smem + (E * T) * 6);                       // [n_kept + 1] first sorted index of every merged row
    int* warp_sum = seg + (E * T) + 4;                                              // [32]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    depend_wait();
    dependents_launch();
    const int n_block_ctas = 2 * a.heads * a.n_blocks * shares;
    const int ch = lane & 7, sub = lane >> 3;   // 16-byte chunk of a row; which of four rows in flight

    if ((int)blockIdx.x >= n_block_ctas) {
        // special tokens: never merged, first in the merged order; T / 8 rows of one head per CTA, all three tensors
        const int idx = blockIdx.x - n_block_ctas, h = idx / sp_chunks, row = (idx % sp_chunks) * (T / 8) + (tid >> 3);
        if (row < a.n_special_total) {
            for (int t = 0; t < 3; ++t) {
                const int m_len = t == 0 ? a.m_q : a.m_k;
                const uint4 v = ld_global(reinterpret_cast<const uint4*>(a.xr[t] + ((int64_t)h * a.n_tokens + row) * kHeadDim) + (tid & 7));
                reinterpret_cast<uint4*>(a.merged[t] + ((int64_t)h * m_len + row) * kHeadDim)[tid & 7] = v;
            }
        }
        return;
    }
    const int per_map = a.heads * a.n_blocks, cta = blockIdx.x / shares, share = blockIdx.x - cta * shares;
    // (the K map, which also merges V, first: its CTAs take longer)
    const int m = 1 - cta / per_map, h = (cta % per_map) / a.n_blocks, b = cta % a.n_blocks;
    const BlockInfo bi = a.blocks[b];
    const int n = bi.n, r = m == 0 ? bi.r_q : bi.r_k, m_len = m == 0 ? a.m_q : a.m_k;
    const bool variable = m == 0 && a.moff_q_var != nullptr;   // after outlier filtering the kept count of a block varies by head
    const int moff = m == 0 ? (variable ? ld_global(a.moff_q_var + (int64_t)h * a.n_blocks + b) : bi.moff_q) : bi.moff_k;
    const int limit = variable ? n : n - r;                    // most kept tokens a valid map can have
    const int64_t base = (int64_t)h * a.n_tokens + bi.start;
    const int32_t* A = a.assign[m] + base;

    const int n_kept = build_groups<T, E>(A, bi.start, n, limit, keys, row_of, seg, warp_sum, nullptr, a.status, m == 0 ? a.rank_q + base : nullptr, moff);
    // eight lanes per merged row (a lane owns one 16-byte chunk of the row), four rows per warp at a time.  The members are
    // taken in position order: the result does not depend on scheduling.
    for (int t = (m == 0 ? 0 : 1); t <= (m == 0 ? 0 : 2); ++t) {
        const __nv_bfloat16* x = a.xr[t] + base * kHeadDim;
        __nv_bfloat16* out = a.merged[t] + ((int64_t)h * m_len + moff) * kHeadDim;
        for (int row = share * (T / 8) + warp * 4 + sub; row < n_kept; row += shares * (T / 8)) {
            const int i0 = seg[row], i1 = seg[row + 1];
            float2 acc[4];
            sum_members(x + 8 * ch, keys, i0, i1, acc);
            if (i1 > i0) {
                const float inv = 1.0f / (float)(i1 - i0);
                uint4 o;
                o.x = pack2(acc[0].x * inv, acc[0].y * inv);
                o.y = pack2(acc[1].x * inv, acc[1].y * inv);
                o.z = pack2(acc[2].x * inv, acc[2].y * inv);
                o.w = pack2(acc[3].x * inv, acc[3].y * inv);
                reinterpret_cast<uint4*>(out + (int64_t)row * kHeadDim)[ch] = o;
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------ outlier filtering
// Query outlier filtering (Sec. 3.4, Algorithm 2) for large blocks: the same steps as for small blocks - deviation of
// every query token from the mean of its group, one threshold over all heads (the refinement kernels of the small-block
// path, which work on the array of deviations), outliers leave their groups - on the sorted group structure of the merge
// kernel.  One CTA per (head, block).

// eps[h][p] = || q_p - mean of the group p was merged into ||_2 in fp32; 0 for a token on its own.
// Bound by the instructions issued and by the gathers (39 warp instructions per token, 61 before; at 40 registers 92 bytes per thread are spilled
// with 8 tokens per thread): two channels per instruction, one exchange for the sums of four
// members and one square root for them took the filter kernels together, at 82 440 tokens x 16 heads in 3840-token blocks, from 221 to 178 us
// (32 976 tokens in 128-token blocks: 104.7 -> 92.2; 137 400 in 64-token blocks: 363 -> 302).
template <int T, int E, bool SHARED>
__global__ void __launch_bounds__(T, kSortedThreads / T) big_deviation_kernel(const OutlierArgs a, int n_shares) {
    const int shares = SHARED ? n_shares : 1;
    extern __shared__ __align__(16) unsigned char mg_smem[];
    uint32_t* keys = reinterpret_cast<uint32_t*>(mg_smem);
    int16_t* row_of = reinterpret_cast<int16_t*>(mg_smem + (E * T) * 4);
    int* seg = reinterpret_cast<int*>(mg_smem + (E * T) * 6);
    int* warp_sum = seg + (E * T) + 4;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ch = lane & 7, sub = lane >> 3;
    const int cta = blockIdx.x / shares, share = blockIdx.x - cta * shares, h = cta / a.n_blocks, b = cta % a.n_blocks;
    const BlockInfo bi = a.blocks[b];
    const int n = bi.n;
    const int64_t base = (int64_t)h * a.n_tokens + bi.start;
    depend_wait();
    dependents_launch();
    float* eps = a.eps + base;
    if (bi.r_q == 0) {   // nothing merged in this block (uniform)
        for (int j = tid; j < n; j += T) eps[j] = 0.f;
        return;
    }
    const int n_kept = build_groups<T, E>(a.assign_q + base, bi.start, n, n, keys, row_of, seg, warp_sum, nullptr, a.status, nullptr, 0);
    const __nv_bfloat16* x = a.src_q.ptr + base * kHeadDim + 8 * ch;   // the reordered copy
    // eight lanes per group (a lane owns 8 of the 64 channels), four groups per warp at a time
    for (int row = share * (T / 8) + warp * 4 + sub; row < ((n_kept + 3) & ~3); row += shares * (T / 8)) {   // (whole sub-groups stay together for the shuffles)
        const bool live = row < n_kept;
        const int i0 = live ? seg[row] : 0, i1 = live ? seg[row + 1] : 0;
        if (i1 - i0 < 2) {
            if (i1 > i0 && ch == 0) eps[keys[i0] & 4095u] = 0.f;
            continue;
        }
        float2 mean[4];
        sum_members(x, keys, i0, i1, mean);
        const float inv = 1.0f / (float)(i1 - i0);
#pragma unroll
        for (int e = 0; e < 4; ++e) mean[e] = make_float2(mean[e].x * inv, mean[e].y * inv);   // kept in fp32
        // (the eight lanes of a group walk its members together: the trip count is the same in all of them); four members
        // at a time, so that four loads are in flight; behind the last member, it again
        const unsigned group_mask = 0xffu << (8 * sub);
        for (int i = i0; i < i1; i += 4) {
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = ld_global(reinterpret_cast<const uint4*>(x + (keys[min(i + u, i1 - 1)] & 4095u) * kHeadDim));
            float d2[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float2 sq = make_float2(0.f, 0.f);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 d = tc::fsub2(unpack2(e == 0 ? v[u].x : e == 1 ? v[u].y : e == 2 ? v[u].z : v[u].w), mean[e]);
                    sq = tc::ffma2(d, d, sq);
                }
                d2[u] = sq.x + sq.y;
            }
            // sums over the eight lanes, each lane ending with one member's: half of them change sides in the first two steps
            const bool b0 = ch & 1, b1 = ch & 2;
            const float o0 = __shfl_xor_sync(group_mask, b0 ? d2[0] : d2[2], 1), o1 = __shfl_xor_sync(group_mask, b0 ? d2[1] : d2[3], 1);
            const float s0 = (b0 ? d2[2] : d2[0]) + o0, s1 = (b0 ? d2[3] : d2[1]) + o1;
            float t = (b1 ? s1 : s0) + __shfl_xor_sync(group_mask, b1 ? s0 : s1, 2);
            t += __shfl_xor_sync(group_mask, t, 4);
            const int at = i + (b0 ? 2 : 0) + (b1 ? 1 : 0);
            if (ch < 4 && at < i1) eps[keys[at] & 4095u] = sqrtf(t);
        }
    }
}

// Outliers (eps > tau) leave their groups: an outlier maps to itself; the other tokens of a group stay together, under
// their old representative if it is not an outlier, else under the remaining member with the lowest position.
template <int T, int E>
__global__ void __launch_bounds__(T, kSortedThreads / T) big_filter_kernel(const OutlierArgs a) {
    extern __shared__ __align__(16) unsigned char mg_smem[];
    uint32_t* keys = reinterpret_cast<uint32_t*>(mg_smem);
    int16_t* row_of = reinterpret_cast<int16_t*>(mg_smem + (E * T) * 4);
    int* seg = reinterpret_cast<int*>(mg_smem + (E * T) * 6);
    int* warp_sum = seg + (E * T) + 4;
    int16_t* rep_of_row = reinterpret_cast<int16_t*>(mg_smem + mg_smem_bytes(E * T));
    unsigned char* outl = mg_smem + mg_smem_bytes(E * T) + (E * T) * 2;
    int16_t* new_rep = reinterpret_cast<int16_t*>(mg_smem + mg_smem_bytes(E * T) + (E * T) * 3);
    __shared__ int s_kept, s_out;
    const int tid = threadIdx.x;
    const int h = blockIdx.x / a.n_blocks, b = blockIdx.x % a.n_blocks;
    const BlockInfo bi = a.blocks[b];
    const int n = bi.n;
    const int64_t base = (int64_t)h * a.n_tokens + bi.start;
    const int32_t* A = a.assign_q + base;
    depend_wait();
    dependents_launch();
    int32_t* A_out = a.assign_q_out + base;
    if (bi.r_q == 0) {   // nothing merged, every deviation is 0: nothing to filter unless everything is an outlier, which changes nothing here
        for (int j = tid; j < n; j += T) A_out[j] = bi.start + j;
        if (tid == 0) a.kept_cnt[(int64_t)h * a.n_blocks + b] = n;
        return;
    }
    if (tid == 0) {
        s_kept = 0;
        s_out = 0;
    }
    const float tau = *a.tau;
    const int n_kept = build_groups<T, E>(A, bi.start, n, n, keys, row_of, seg, warp_sum, rep_of_row, a.status, nullptr, 0);
    int n_out = 0;
    for (int j = tid; j < n; j += T) {
        const bool o = a.eps[base + j] > tau;
        outl[j] = o ? 1 : 0;
        n_out += o ? 1 : 0;
    }
    __syncthreads();
    for (int row = tid; row < n_kept; row += T) {   // a thread per group: groups are short, the rare long one costs its thread a scan
        const int rp = rep_of_row[row];
        int nr = rp;
        if (outl[rp]) {
            nr = -1;
            for (int i = seg[row]; i < seg[row + 1]; ++i) {
                const int pos = (int)(keys[i] & 4095u);
                if (!outl[pos]) {
                    nr = pos;
                    break;
                }
            }
        }
        new_rep[row] = (int16_t)nr;
    }
    __syncthreads();
    int kept = 0;
    for (int j = tid; j < n; j += T) {
        int target = j;
        if (!outl[j]) {
            int rp = A[j] - bi.start;
            if (rp < 0 || rp >= n) rp = j;                  // (recorded by build_groups)
            const int row = row_of[rp];
            if (row >= 0 && row < n_kept) target = new_rep[row];   // never -1 here: j itself is a remaining member
            if (target < 0) target = j;
        }
        A_out[j] = bi.start + target;
        kept += target == j ? 1 : 0;
    }
    atomicAdd(&s_kept, kept);
    atomicAdd(&s_out, n_out);
    __syncthreads();
    if (tid == 0) {
        a.kept_cnt[(int64_t)h * a.n_blocks + b] = s_kept;
        if (s_out) atomicAdd(a.sel + kSelOutliers, s_out);
    }
}

}  // namespace

// threads per CTA and tokens per thread for blocks of up to max_block tokens
template <typename F>
cudaError_t with_cta_size(int max_block, F&& f) {
    using four = std::integral_constant<int, 4>;
    if (max_block <= 256) return f(std::integral_constant<int, 64>{}, four{});
    if (max_block <= 512) return f(std::integral_constant<int, 128>{}, four{});
    if (max_block <= 1024) return f(std::integral_constant<int, 256>{}, four{});
    if (max_block <= 2048) return f(std::integral_constant<int, 512>{}, four{});
    return f(std::integral_constant<int, 512>{}, std::integral_constant<int, 8>{});
}

// CTAs for a block of the kernels that sort its tokens and then gather the rows of its groups, where blocks alone would leave SMs without: each sorts all tokens and
// gathers a share of the rows: merge of 64 maps of up to 1408 tokens 23.6 -> 17.4 us, of 96 of up to 1024 29.7 -> 19.5.  (With more of them than fit at once every
// sort is paid for: two CTAs for each of 704 maps of 3840 tokens 225 -> 250 us.)
int row_shares(int64_t blocks, int64_t resident) {
    const int64_t s = resident / (blocks > 0 ? blocks : 1);
    return (int)(s < 1 ? 1 : s > 4 ? 4 : s);
}

cudaError_t launch_big_deviation(const OutlierArgs& a, int max_block, int sm_count, cudaStream_t stream) {
    return with_cta_size(max_block, [&](auto t, auto e) {
        constexpr int T = decltype(t)::value, E = decltype(e)::value;
        const int shares = row_shares((int64_t)a.heads * a.n_blocks, (int64_t)(kSortedThreads / T) * sm_count);
        return launch_kernel(shares > 1 ? big_deviation_kernel<T, E, true> : big_deviation_kernel<T, E, false>, a.heads * a.n_blocks * shares, T, mg_smem_bytes(E * T), stream, a, shares);
    });
}

cudaError_t launch_big_filter(const OutlierArgs& a, int max_block, cudaStream_t stream) {
    return with_cta_size(max_block, [&](auto t, auto e) {
        constexpr int T = decltype(t)::value, E = decltype(e)::value;
        return launch_kernel(big_filter_kernel<T, E>, a.heads * a.n_blocks, T, of_smem_bytes(E * T), stream, a);
    });
}

template <int T, int E>
cudaError_t configure_sorted_group_kernels() {
    cudaError_t e = cudaSuccess;
    auto set = [&](auto kernel, int bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    set(big_merge_kernel<T, E, false>, mg_smem_bytes(E * T));
    set(big_merge_kernel<T, E, true>, mg_smem_bytes(E * T));
    set(big_deviation_kernel<T, E, false>, mg_smem_bytes(E * T));
    set(big_deviation_kernel<T, E, true>, mg_smem_bytes(E * T));
    set(big_filter_kernel<T, E>, of_smem_bytes(E * T));
    return e;
}

cudaError_t configure_big_blocks() {
    // setmaxnreg.inc takes registers from those the CTA was launched with, and waits without limit for more than there are
    cudaError_t e = cudaSuccess;
    for (auto scores : {big_scores_kernel<false>, big_scores_kernel<true>}) {
        cudaFuncAttributes launched;
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&launched, scores);
        if (e == cudaSuccess && launched.numRegs * SC_THREADS < 128 * kScoreRoleRegs + (SC_THREADS - 128) * kScoreMaxRegs) e = cudaErrorInvalidConfiguration;
        if (e == cudaSuccess) e = cudaFuncSetAttribute(scores, cudaFuncAttributeMaxDynamicSharedMemorySize, SC_SMEM);
    }
    if (e == cudaSuccess) e = configure_sorted_group_kernels<64, 4>();
    if (e == cudaSuccess) e = configure_sorted_group_kernels<128, 4>();
    if (e == cudaSuccess) e = configure_sorted_group_kernels<256, 4>();
    if (e == cudaSuccess) e = configure_sorted_group_kernels<512, 4>();
    if (e == cudaSuccess) e = configure_sorted_group_kernels<512, 8>();
    return e;
}

cudaError_t launch_big_scores(const BigMatchArgs& args, int sm_count, cudaStream_t stream) {
    // Where there are fewer blocks than SMs their src tokens are shared out: every part copies all dst tokens (about 6 us), so only for SMs that have nothing else to do.
    // 64 items of up to 1408 tokens 31.6 -> 25.5 us.
    BigMatchArgs a = args;
    const int64_t blocks = 2ll * a.heads * a.n_blocks;
    const int sms = sm_count < 1 ? 1 : sm_count;
    a.parts = (int)(blocks < 1 || blocks > sms ? 1 : sms / blocks > 4 ? 4 : sms / blocks);
    const int64_t total = blocks * a.parts;
    const int ctas = (int)(total > sms ? sms : total < 1 ? 1 : total);
    return launch_kernel(a.parts > 1 ? big_scores_kernel<true> : big_scores_kernel<false>, ctas, SC_THREADS, SC_SMEM, stream, a);
}

cudaError_t launch_big_select(const BigMatchArgs& a, cudaStream_t stream) {
    return launch_kernel(big_select_kernel, 2 * a.heads * a.n_blocks, SEL_THREADS, 0, stream, a);
}

cudaError_t launch_big_merge(const MergeArgs& a, int max_block, int sm_count, cudaStream_t stream) {
    return with_cta_size(max_block, [&](auto t, auto e) {
        constexpr int T = decltype(t)::value, E = decltype(e)::value;
        const int sp_chunks = (a.n_special_total + T / 8 - 1) / (T / 8);
        const int shares = row_shares(2ll * a.heads * a.n_blocks, (int64_t)(kMergeThreads / T) * sm_count);
        return launch_kernel(shares > 1 ? big_merge_kernel<T, E, true> : big_merge_kernel<T, E, false>, 2 * a.heads * a.n_blocks * shares + a.heads * sp_chunks, T, mg_smem_bytes(E * T), stream, a, sp_chunks, shares);
    });
}

}  // namespace httm
