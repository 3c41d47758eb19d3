// Matching and merging for merging blocks of at most 32 tokens (Eq. 1, Sec. 3.2), one warp per UNIT = one (head, block) with all
// its tensors: the match kernel works off Q and K of a block, the merge kernel Q, K and V (V follows K's map).
// Blocks of up to 64 tokens are matched here too.
//
// A block is 4 KB and 5 KFLOP per tensor, so what bounds these kernels is not the arithmetic but the instructions around it:
// table entries, block geometry, dst positions, the next load.  With one task per (tensor, head, block) the match kernel
// issued 697 warp instructions per task and the merge kernel 575, at 50 - 56 % of the issue slots with 16 warps per SM.  Here
//   - table entry, geometry and cursor are taken once per unit, one unit ahead;
//   - what a lane needs to know about a block's shape (which rows hold its dst tokens, which tokens it owns) is kept from block
//     to block and recomputed when the shape changes (clipped blocks at the edges of the grid);
//   - K's groups serve V, and the maps are read once per unit;
//   - results leave through the stage as whole rows instead of 4 bytes per lane.
// Measured at 32 976 tokens x 16 heads, 32-token blocks: match 53 -> 39.6 us, merge 69.6 -> 62.4 us (both
// with the interval between two events).  What is left is the latency of a warp's instruction stream, hence as few instructions as possible
// (match: one token per lane from the arg-max on) and as many warps as fit (merge: two stages).
#include "httm_blocks.cuh"
#include "httm_launch.cuh"

#include <math_constants.h>

namespace httm {

namespace {

constexpr int kWarps = 8;
constexpr uint32_t kStage = 32 * kRowBytes;   // one block of one tensor, 128-byte swizzle

// ------------------------------------------------------------------------------------ match
// Per tensor: cosine of every token with every dst token (at most 8), best dst per src token, the r best src tokens
// merge; ties go to the lowest dst and the lowest src position.  The dot products and the squared norms (diagonals of a tile
// against itself) are m16n8k16 MMAs on ldmatrix fragments of the swizzled stage; the dst rows are gathered by giving
// ldmatrix their addresses.  Products of bf16 values are exact in fp32.
// (Every lane owns one token when the r best are chosen.  With two tokens in every other lane a tensor took 518 instructions, now 441, and the kernel alone, one launch
// at a time, 39.3 -> 34.8 us at 32 976 tokens; between the other kernels of a call 40.8 -> 40.4, 65 952 tokens 82.9 -> 72.7.)
// Row rho of the stage is owned, from the arg-max on, by lane (rho & 7) * 4 + (rho >> 3).
constexpr int kMatchSmem = kWarps * (2 * (int)kStage + 16) + 1024 /*alignment slack*/;   // two blocks of 32 rows or one of 64 per warp

constexpr int match_ctas(int tiles) { return tiles == 2 ? 3 : 2; }   // per SM: 80 registers (with whole units 72 bytes of them spilled) and 120
// TILES: blocks of up to 32 tokens, 8 dst tokens (2); or up to 64 tokens, 16 dst tokens (4), where a warp has room for one tensor, so that 16 warps fit on an SM.
// UNITS: a task is a unit, both its tensors in a stage each; else one tensor of it.  ONE: no warp has a second task, and nothing for the next one is kept or looked up:
// calls in 32-token blocks on 1 044 tokens x 16 heads 18.0 -> 17.6 us, 2 219 x 16 23.6 -> 23.1, 2 219 x 8 21.4 -> 20.4; 48-token blocks, 1 167 x 8 20.4 -> 20.2.
// A team of one warp that kept all fragments of a 64-token block and had two stages, of which 10 fitted on an SM, both tensors of a unit in turn through one stage, and a
// tensor at a time: 137 400 tokens x 16 heads in 64-token blocks, ratio 0.8, match 166.2 / 137.5 / 131.5 us; calls on 16 488 tokens 113.7 / 115.7 / 111.4 (4800 units on 2368
// warps: three rounds of units, five of tensors), on 10 992 tokens 67.1 / 68.2 / 64.6; 7 898 tokens in 48-token blocks 93.1 / 92.7 / 90.7.  (24 warps with 80 registers spill.)
template <int TILES, bool DIRECT, bool UNITS, bool ONE>
__global__ void __launch_bounds__(kWarps * 32, match_ctas(TILES))
match_small_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ MatchArgs a) {
    constexpr int ND = TILES / 2, SLOTS = TILES / 2;   // groups of eight dst tokens; tokens per lane
    constexpr int STAGES = UNITS ? 2 : 1;
    static_assert(!UNITS || (TILES == 2 && !ONE), "a warp has room for two tensors of 32 tokens; few units are dealt out as tensors");
    constexpr uint32_t STAGE = TILES * 16 * kRowBytes;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + align_pad(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tq = lane & 3;   // accumulator layout: rows g, g + 8; columns 2 tq, 2 tq + 1
    const int rho0 = 8 * tq + g;               // the stage rows this lane owns: rho0 + 32 i
    const uint32_t stage0 = smem_u32(smem + (size_t)warp * 2 * kStage);
    const uint32_t bar0 = smem_u32(smem + (size_t)kWarps * 2 * kStage + warp * 16);
    if (lane == 0) {
        mbar_init(bar0, 1);
        mbar_init(bar0 + 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();

    Box box{};
    if (DIRECT) box.set(a.layout);
    const int64_t n_tasks = (UNITS ? 1ll : 2ll) * a.heads * a.n_blocks;
    const int stride = gridDim.x * kWarps, first = blockIdx.x * kWarps + warp;
    UnitCursor next;   // the task whose loads are issued next; a tensor at a time: K's heads follow Q's
    next.init(first, stride, a.n_blocks);
    auto issue = [&](int t, uint32_t st, const int4& geom, int start, int h) {   // lane 0 only
        const Geometry bg = unpack_geometry(geom);
        const uint32_t mb = bar0 + 8 * st;
        const CUtensorMap* m = t == 0 ? &map_q : &map_k;
        if (DIRECT) {
            mbar_expect_tx(mb, (uint32_t)box.rows * kRowBytes);
            tma_block_load(stage0 + st * STAGE, m, mb, bg.x0, bg.y0, bg.s0, h);
        } else {
            mbar_expect_tx(mb, STAGE);
            tma_rows_load(stage0 + st * STAGE, m, mb, start, h);
        }
    };
    BlockInfo bi_next{};
    int4 bg_next{};
    int h_next = 0, t_next = 0;   // (t_next: first tensor of the task)
    auto fetch = [&]() {
        bi_next = a.blocks[next.u];
        if (DIRECT) bg_next = load_geometry(a.geom, next.u);
        t_next = !UNITS && next.h >= a.heads ? 1 : 0;
        h_next = next.h - t_next * a.heads;
    };
    if (first < n_tasks) fetch();
    depend_wait();
    dependents_launch();
    clear_words(a.clear, blockIdx.x, gridDim.x);
    if (first < n_tasks && lane == 0)
        for (int st = 0; st < STAGES; ++st) issue(t_next + st, st, bg_next, bi_next.start, h_next);

    // ldmatrix offsets of a 16-row tile: rows 0-7 / 8-15 (lane bit 3), k chunk 2 ks / 2 ks + 1 (lane bit 4); chunk c of row j sits at c ^ (j & 7)
    uint32_t a_off[4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) a_off[ks] = ((lane & 7) + ((lane >> 3) & 1) * 8) * kRowBytes + (((2 * ks + (lane >> 4)) ^ (lane & 7)) << 4);
    // what this lane knows about the shape of the blocks at hand
    int shape_a = -1, shape_b = -1;
    uint32_t d_off[ND][2];        // ldmatrix offsets of dst rows 8 d + (lane & 7)
    int d_pos = 0;                // token number of dst lane & (8 ND - 1)
    int tok[SLOTS];               // tokens owned (-1: none)
    bool is_src[SLOTS];
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) {
        d_off[i][0] = d_off[i][1] = 0;
        tok[i] = -1;
        is_src[i] = false;
    }

    uint32_t seq = 0;   // tensors so far: in stage seq % STAGES
    bool failed = false, ahead = false;   // ahead: the next tensor's load is in flight too
    for (int64_t task = first; task < n_tasks; task += stride) {
        const BlockInfo bi = bi_next;
        const int4 geom = bg_next;
        const int h = h_next, t0 = t_next, n = bi.n;
        const bool more = !ONE && task + stride < n_tasks;
        if (more) {
            next.advance();
            fetch();   // in flight while this task is worked off
        }
#pragma unroll 1
        for (int t = t0; t < t0 + STAGES; ++t, ++seq) {
            const uint32_t st = seq % STAGES;
            auto refill = [&]() {   // the tensor that takes this stage next (lane 0 only)
                if (more) issue(UNITS ? t : t_next, st, bg_next, bi_next.start, h_next);
            };
            const int r = t == 0 ? bi.r_q : bi.r_k, nd = t == 0 ? bi.nd_q : bi.nd_k;
            int32_t* A = a.assign[t] + (int64_t)h * a.n_tokens + bi.start;
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar0 + 8 * st, seq / STAGES & 1u, a.status, kDevTimeoutMatchLoad))) {
                failed = true;
                ahead = UNITS && (t < 1 || more);
                break;
            }
            if (r == 0 || nd > 8 * ND) {   // nothing merges, or an anchored block with more dst tokens (match_anchor_kernel)
                if (r == 0)
                    for (int j = lane; j < n; j += 32) A[j] = bi.start + j;
                __syncwarp();
                if (lane == 0) refill();
                continue;
            }
            const int n_rows = DIRECT ? box.rows : n;   // rows of the stage that may hold tokens
            {
                const int sa = n | (nd << 8) | (bi.n_rule << 16), sb = DIRECT ? shape_key(geom) : 0;   // (n and n_rule at most 64)
                if (sa != shape_a || sb != shape_b) {
                    const Geometry bg = unpack_geometry(geom);
                    shape_a = sa;
                    shape_b = sb;
                    const int n_rule = bi.n_rule;   // n (evenly spaced dst tokens) or n_dst (the first n_dst tokens: first-frame anchoring)
                    d_pos = small_div((min(lane & (8 * ND - 1), nd - 1) + 1) * n_rule + nd - 1, nd) - 1;
#pragma unroll
                    for (int d = 0; d < ND; ++d) {
                        const int pos = ND == 1 ? d_pos : __shfl_sync(0xffffffffu, d_pos, 8 * d + (lane & 7)), row = DIRECT ? row_of_token(box, bg, pos) : pos;
#pragma unroll
                        for (int kp = 0; kp < 2; ++kp) d_off[d][kp] = row * kRowBytes + (((4 * kp + (lane >> 3)) ^ (row & 7)) << 4);
                    }
#pragma unroll
                    for (int i = 0; i < SLOTS; ++i) {
                        const int rho = rho0 + 32 * i, j = DIRECT ? token_of_row(box, bg, rho) : (rho < n ? rho : -1);
                        tok[i] = j;
                        is_src[i] = j >= 0 && !(j < n_rule && small_div((j + 1) * nd, n_rule) > small_div(j * nd, n_rule));
                    }
                }
            }
            const uint32_t blk = stage0 + st * STAGE;
            // ---- dst fragments (k steps 2 kp, 2 kp + 1 per ldmatrix.x4) and their norms: lane 9 tq holds that of dst 2 tq, 9 tq + 4 of 2 tq + 1
            uint32_t bf[ND][4][2];
            float w0[ND], w1[ND];
#pragma unroll
            for (int d = 0; d < ND; ++d) {
                w0[d] = w1[d] = CUDART_NAN_F;
                if (d == 0 || 8 * d < nd) {   // (uniform)
#pragma unroll
                    for (int kp = 0; kp < 2; ++kp) {
                        uint32_t rr[4];
                        ldmatrix_x4(rr, blk + d_off[d][kp]);
                        bf[d][2 * kp][0] = rr[0];
                        bf[d][2 * kp][1] = rr[1];
                        bf[d][2 * kp + 1][0] = rr[2];
                        bf[d][2 * kp + 1][1] = rr[3];
                    }
                    float dn[4];
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        const uint32_t ad[4] = {bf[d][ks][0], bf[d][ks][0], bf[d][ks][1], bf[d][ks][1]};
                        if (ks == 0)
                            mma_first(dn, ad, bf[d][ks][0], bf[d][ks][1]);
                        else
                            mma_bf16_16816(dn, ad, bf[d][ks][0], bf[d][ks][1]);
                    }
                    const float dsel = (g & 1) ? dn[1] : dn[0];
                    w0[d] = inv_norm(__shfl_sync(0xffffffffu, dsel, 9 * tq));
                    w1[d] = inv_norm(__shfl_sync(0xffffffffu, dsel, 9 * tq + 4));
                    if (8 * d + 2 * tq >= nd) w0[d] = CUDART_NAN_F;
                    if (8 * d + 2 * tq + 1 >= nd) w1[d] = CUDART_NAN_F;
                }
            }
            // ---- best dst of every row.  The four lanes of a row meet: an exchange with lane ^ 1 leaves a lane one of a tile's rows g and g + 8, one with
            // lane ^ 2 one of the two tiles
            const bool odd = tq & 1, high = tq & 2;
            auto meet = [](float& top, int& arg, float send, int send_arg, int with) {
                const float ov = __shfl_xor_sync(0xffffffffu, send, with);
                const int oa = __shfl_xor_sync(0xffffffffu, send_arg, with);
                if (ov > top || (ov == top && oa < arg)) {   // (ties: the lower dst)
                    top = ov;
                    arg = oa;
                }
            };
            float top[TILES], norm[TILES];
            int arg[TILES];
#pragma unroll
            for (int mt = 0; mt < TILES; ++mt) {
                top[mt] = -INFINITY;
                norm[mt] = 0.f;
                arg[mt] = 0;
                if (mt * 16 < n_rows) {   // warp-uniform
                    float c[ND][4], lo[4], hi[4];
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        uint32_t af[4];
                        ldmatrix_x4(af, blk + mt * 16 * kRowBytes + a_off[ks]);
                        if (ks == 0) {
#pragma unroll
                            for (int d = 0; d < ND; ++d)
                                if (d == 0 || 8 * d < nd) mma_first(c[d], af, bf[d][ks][0], bf[d][ks][1]);
                            mma_first(lo, af, af[0], af[2]);   // against rows 0-7 of the tile
                            mma_first(hi, af, af[1], af[3]);   // against rows 8-15
                        } else {
#pragma unroll
                            for (int d = 0; d < ND; ++d)
                                if (d == 0 || 8 * d < nd) mma_bf16_16816(c[d], af, bf[d][ks][0], bf[d][ks][1]);
                            mma_bf16_16816(lo, af, af[0], af[2]);
                            mma_bf16_16816(hi, af, af[1], af[3]);
                        }
                    }
                    // this lane's dst tokens first, for rows g and g + 8
                    // (the maximum with -infinity drops what is not a number: a place without a dst token, tokens whose norm overflows)
                    float t0 = 0.f, t1 = 0.f;
                    int d0 = 0, d1 = 0;
#pragma unroll
                    for (int d = 0; d < ND; ++d) {
                        if (d == 0 || 8 * d < nd) {
                            const float s00 = fmaxf(c[d][0] * w0[d], -INFINITY), s01 = fmaxf(c[d][1] * w1[d], -INFINITY);
                            const float s10 = fmaxf(c[d][2] * w0[d], -INFINITY), s11 = fmaxf(c[d][3] * w1[d], -INFINITY);
                            const float u0 = fmaxf(s00, s01), u1 = fmaxf(s10, s11);
                            const int e0 = 8 * d + 2 * tq + (s01 > s00 ? 1 : 0), e1 = 8 * d + 2 * tq + (s11 > s10 ? 1 : 0);
                            if (d == 0 || u0 > t0) {
                                t0 = u0;
                                d0 = e0;
                            }
                            if (d == 0 || u1 > t1) {
                                t1 = u1;
                                d1 = e1;
                            }
                        }
                    }
                    top[mt] = odd ? t1 : t0;
                    arg[mt] = odd ? d1 : d0;
                    meet(top[mt], arg[mt], odd ? t0 : t1, odd ? d0 : d1, 1);
                    const int diag = 4 * g + (g >> 1);   // the lane that holds the squared norms of rows g and g + 8
                    const float nl = __shfl_sync(0xffffffffu, (g & 1) ? lo[1] : lo[0], diag), nh = __shfl_sync(0xffffffffu, (g & 1) ? hi[3] : hi[2], diag);
                    norm[mt] = odd ? nh : nl;
                }
            }
            uint32_t key[SLOTS];   // 0: not a src token
            int best[SLOTS];
#pragma unroll
            for (int i = 0; i < SLOTS; ++i) {
                float best_score = high ? top[2 * i + 1] : top[2 * i];
                best[i] = high ? arg[2 * i + 1] : arg[2 * i];
                meet(best_score, best[i], high ? top[2 * i] : top[2 * i + 1], high ? arg[2 * i] : arg[2 * i + 1], 2);
                key[i] = is_src[i] ? score_key(best_score * inv_norm(high ? norm[2 * i + 1] : norm[2 * i])) : 0u;
            }
            __syncwarp();   // every lane has read the stage
            if (lane == 0) refill();

            // ---- the r src with the best scores merge (ties: lowest position first)
            const int n_out = n - nd - r;
            bool merged[SLOTS];
            if (r <= n_out) {
#pragma unroll
                for (int i = 0; i < SLOTS; ++i) merged[i] = false;
                for (int round = 0; round < r; ++round) {
                    uint32_t k[SLOTS], top_key = 0u;
#pragma unroll
                    for (int i = 0; i < SLOTS; ++i) {
                        k[i] = merged[i] ? 0u : key[i];
                        top_key = max(top_key, k[i]);
                    }
                    top_key = __reduce_max_sync(0xffffffffu, top_key);
                    unsigned at = 0xffffffffu;
#pragma unroll
                    for (int i = SLOTS - 1; i >= 0; --i)
                        if (k[i] == top_key) at = rho0 + 32 * i;
                    const unsigned win = __reduce_min_sync(0xffffffffu, at);   // lowest position holding it
#pragma unroll
                    for (int i = 0; i < SLOTS; ++i) merged[i] = merged[i] || (is_src[i] && win == (unsigned)(rho0 + 32 * i));
                }
            } else {
#pragma unroll
                for (int i = 0; i < SLOTS; ++i) merged[i] = is_src[i];
                for (int round = 0; round < n_out; ++round) {
                    uint32_t low = 0xffffffffu;
#pragma unroll
                    for (int i = 0; i < SLOTS; ++i) low = min(low, merged[i] ? key[i] : 0xffffffffu);
                    low = __reduce_min_sync(0xffffffffu, low);
                    int at = -1;
#pragma unroll
                    for (int i = 0; i < SLOTS; ++i)
                        if (merged[i] && key[i] == low) at = rho0 + 32 * i;
                    const int win = __reduce_max_sync(0xffffffffu, at);   // highest position
#pragma unroll
                    for (int i = 0; i < SLOTS; ++i) merged[i] = merged[i] && win != rho0 + 32 * i;
                }
            }
#pragma unroll
            for (int i = 0; i < SLOTS; ++i) {
                const int target = __shfl_sync(0xffffffffu, d_pos, best[i]);
                if (tok[i] >= 0) A[tok[i]] = bi.start + (merged[i] ? target : tok[i]);
            }
        }
        if (failed) break;
        if (ONE) break;
    }
    if (failed)   // give copies that may still be in flight a bounded chance to land before the shared memory is released
        for (uint32_t i = seq; i <= seq + (ahead ? 1 : 0); ++i) mbar_wait_bounded(bar0 + 8 * (i % STAGES), i / STAGES & 1u, a.status, kDevTimeoutMatchLoad);
}

// ------------------------------------------------------------------------------------ merge
// The group sums of a block are one small dense contraction: merged_sum[kept row][channel] = sum_token W[row][token] x[token][channel]
// with the 0/1 assignment matrix W (exact in bf16, built in registers from the map), fp32 accumulation, times the reciprocal
// of the group size, one rounding to bf16.  Kept tokens are compacted in reordered order.  The rows go through the stage they came
// from, 16 channels at a time (whose fragments are in registers by then), and leave 16 bytes per lane, whole rows; then the stage is refilled.
// Tensor i of the warp's sequence Q K V Q K V .. lies in stage i & 1.  With a stage for each tensor and all 64 channels in registers at a time (128 of them) 16 warps
// were all that fits on an SM: 61.4 -> 57.3 us at 32 976 tokens, 132 -> 115 at 65 952, 19.5 -> 17.5 at 5 516 (unit_ctas).
constexpr int kMergeAux = 32 * 4 + 32 * 4 + 16 + 64;   // reciprocal group sizes, group sizes, 2 mbarriers, merged rows of the tokens
constexpr int kMergeStages = 2;
constexpr int kMergeSmem = kWarps * (kMergeStages * (int)kStage + kMergeAux) + 1024 /*alignment slack*/;

__device__ __forceinline__ void stmatrix_x4(uint32_t saddr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(saddr), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}
template <int CTAS, bool DIRECT, bool SPLIT>   // CTAS: per SM
__global__ void __launch_bounds__(kWarps * 32, CTAS) merge_small_kernel(const __grid_constant__ MergeMaps maps, const __grid_constant__ MergeArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + align_pad(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tq = lane & 3;   // accumulator layout: rows g, g + 8; columns 2 tq, 2 tq + 1
    unsigned char* stage = smem + warp * (kMergeStages * kStage);
    unsigned char* aux = smem + kWarps * kMergeStages * kStage + warp * kMergeAux;
    float* rcnt = reinterpret_cast<float*>(aux);             // [32] 1 / group size of kept row
    int* gsz = reinterpret_cast<int*>(aux + 32 * 4);         // [32] size of kept row
    const uint32_t stage0 = smem_u32(stage), bar0 = smem_u32(aux + 2 * 32 * 4);
    __nv_bfloat16* rows_of = reinterpret_cast<__nv_bfloat16*>(aux + 2 * 32 * 4 + 16);   // [32] merged rows of the tokens, in fragment order
    if (lane == 0) {
#pragma unroll
        for (int st = 0; st < kMergeStages; ++st) mbar_init(bar0 + 8 * st, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    Box box{};
    if (DIRECT) box.set(a.layout);
    const int own_t = DIRECT ? lane / (box.h * box.w) : 0, own_y = DIRECT ? (lane / box.w) % box.h : 0, own_x = DIRECT ? lane % box.w : 0;
    if (DIRECT)   // stage rows that no block load writes enter the MMAs with weight 0: they must hold finite values
        for (int q = box.rows * 8 + lane; q < 32 * 8; q += 32)
#pragma unroll
            for (int st = 0; st < kMergeStages; ++st) *reinterpret_cast<uint4*>(stage + st * kStage + q * 16) = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();

    // units 0 .. n_blocks - 1 of a head are merging blocks, the rest special tokens (never merged: copied)
    const int sp_units = DIRECT ? (a.layout.n_special > 0 ? a.layout.frames : 0) : (a.n_special_total + 31) / 32;
    const int per_head = a.n_blocks + sp_units;
    const int64_t n_units = (int64_t)a.heads * per_head;
    int stride = gridDim.x * kWarps, first = blockIdx.x * kWarps + warp, t_first = 0, t_last = 2;
    if (SPLIT) {
        t_first = t_last = (int)min((int64_t)2, first / n_units);
        first = (int)min(n_units, first - t_first * n_units);
        stride = (int)n_units;
    }
    struct Meta {
        int h, start, sizes, moff_q, moff_k;   // sizes: n | r_q << 8 | r_k << 16, bit 24: special tokens
        int4 geom;                             // (of special tokens: .w = their frame)
        __device__ int n() const { return sizes & 0xff; }
        __device__ int r(int t) const { return (sizes >> (t == 0 ? 8 : 16)) & 0xff; }
        __device__ bool special() const { return sizes >> 24; }
    };
    UnitCursor next;
    next.init(first, stride, per_head);
    auto fetch = [&]() {
        Meta m{};
        m.h = next.h;
        if (next.u >= a.n_blocks) {
            m.geom.w = next.u - a.n_blocks;
            m.start = m.geom.w * (DIRECT ? a.layout.n_special : 32);
            m.sizes = (1 << 24) | (DIRECT ? a.layout.n_special : min(32, a.n_special_total - m.start));
            m.moff_q = m.moff_k = m.start;
        } else {
            if (DIRECT) m.geom = load_geometry(a.geom, next.u);
            const BlockInfo bi = a.blocks[next.u];
            m.start = bi.start;
            m.sizes = bi.n | (bi.r_q << 8) | (bi.r_k << 16);
            m.moff_q = bi.moff_q;
            m.moff_k = bi.moff_k;
        }
        return m;
    };
    auto fetch_offset = [&](Meta* m) {   // with outlier filtering the heads' rows start elsewhere
        if (a.moff_q_var && next.u < a.n_blocks) m->moff_q = ld_global(a.moff_q_var + (int64_t)m->h * a.n_blocks + next.u);
    };
    auto issue = [&](int t, uint32_t st, const Meta& m) {   // lane 0 only
        const uint32_t mb = bar0 + 8 * st, dst = stage0 + st * kStage;
        if (!DIRECT) {
            mbar_expect_tx(mb, kStage);   // (rows past the head's end are zero filled)
            tma_rows_load(dst, &maps.block[t], mb, m.start, m.h);
        } else if (m.special()) {
            mbar_expect_tx(mb, (uint32_t)m.n() * kRowBytes);
            asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
                         "l"(reinterpret_cast<uint64_t>(&maps.special[t])), "r"(mb), "r"(0), "r"(0), "r"(m.geom.w), "r"(m.h)
                         : "memory");
        } else {
            const Geometry bg = unpack_geometry(m.geom);
            mbar_expect_tx(mb, (uint32_t)box.rows * kRowBytes);
            tma_block_load(dst, &maps.block[t], mb, bg.x0, bg.y0, bg.s0, m.h);
        }
    };
    // lane = row of the stage; number of the token it holds in the block (-1: none)
    auto token_of_lane = [&](const Meta& m) {
        if (!DIRECT || m.special()) return lane < m.n() ? lane : -1;
        const Geometry bg = unpack_geometry(m.geom);
        return own_t < bg.frames && own_y < bg.rows && own_x < bg.cols ? (own_t * bg.rows + own_y) * bg.cols + own_x : -1;
    };
    auto load_target = [&](const Meta& m, int map) {   // token this lane's token is merged into (number in the block)
        const int tok = token_of_lane(m);
        return m.r(map) > 0 && tok >= 0 ? ld_global(a.assign[map] + (int64_t)m.h * a.n_tokens + m.start + tok) - m.start : -1;
    };
    Meta meta_next{};
    if (first < n_units) meta_next = fetch();
    auto issue_first = [&]() {
        if (first < n_units && lane == 0)
#pragma unroll
            for (int i = 0; i < (SPLIT ? 1 : 2); ++i) issue(t_first + i, i, meta_next);
    };
    if (a.early) issue_first();
    depend_wait();
    dependents_launch();
    if (!a.early) issue_first();
    int target_next[2] = {-1, -1};
    if (first < n_units) {
        fetch_offset(&meta_next);
        if (t_first == 0) target_next[0] = load_target(meta_next, 0);
        if (t_last > 0) target_next[1] = load_target(meta_next, 1);
    }

    const float recip = 1.0f / (float)(lane + 1);   // lane i holds 1 / (i + 1)

    uint32_t seq = 0;   // tensors so far: in stage seq & 1
    bool failed = false, ahead = false;   // ahead: the next tensor's load is in flight too
    for (int64_t unit = first; unit < n_units; unit += stride) {
        const Meta m = meta_next;
        const int target[2] = {target_next[0], target_next[1]};
        const bool more = unit + stride < n_units;
        if (more) {
            next.advance();
            meta_next = fetch();   // in flight while this unit is worked off
            fetch_offset(&meta_next);
        }
        const int tok = token_of_lane(m), n = m.n();
        uint32_t af0[2][4];   // W fragments of the first 16 merged rows (K's serve V)
        const int n_ks = (DIRECT ? box.rows : n) > 16 ? 2 : 1;   // 16-row steps of the stage that may hold tokens
        int row_of = -1, n_kept = 0;
        uint2 rw[2];
#pragma unroll 1
        for (int t = SPLIT ? t_first : 0; t <= (SPLIT ? t_last : 2); ++t, ++seq) {
            const uint32_t st = seq & 1u;
            const int r = m.r(t), moff = t == 0 ? m.moff_q : m.moff_k, m_len = t == 0 ? a.m_q : a.m_k;
            uint4* out = reinterpret_cast<uint4*>(a.merged[t] + ((int64_t)m.h * m_len + moff) * kHeadDim);
            const uint32_t blk = stage0 + st * kStage;
            const unsigned char* rows = stage + st * kStage;
            int n_out = n;   // rows that leave
            if (r > 0 && (SPLIT || t < 2)) {   // the groups of this map (V follows K)
                int rep = t == 0 ? target[0] : target[1];
                if (tok >= 0) {
                    if (rep < 0 || rep >= n) {   // corrupt map: record, treat as kept
                        atomicCAS(a.status, kDevOk, kDevBadIndex);
                        rep = tok;
                    }
                    if (DIRECT) rep = row_of_token(box, unpack_geometry(m.geom), rep);   // ROW of the stage holding the token it is merged into
                } else {
                    rep = -1;
                }
                // merged row of every token: rank of its representative among the kept tokens
                const unsigned kept = __ballot_sync(0xffffffffu, rep == lane);
                n_kept = __popc(kept);
                row_of = rep >= 0 ? __popc(kept & ((1u << rep) - 1u)) : -1;
                gsz[lane] = 0;
                __syncwarp();
                rows_of[fragment_order(lane)] = __float2bfloat16_rn((float)row_of);
                const int slot = row_of >= 0 ? atomicAdd(&gsz[row_of], 1) : 0;   // (the order of a row's members does not matter)
                __syncwarp();
                const int sz = gsz[lane];
                rcnt[lane] = __shfl_sync(0xffffffffu, recip, (sz - 1) & 31);
                __syncwarp();
                if (t == 0) {
                    if (tok >= 0) a.rank_q[(int64_t)m.h * a.n_tokens + m.start + tok] = moff + row_of;
                    if (a.group_start) {
                        // member lists of the merged rows: the block's tokens group by group, kept rows in rank order
                        // (first member of row k = tokens of the rows before it: a warp scan over the group sizes)
                        int incl = sz;
#pragma unroll
                        for (int off = 1; off < 32; off <<= 1) {
                            const int v = __shfl_up_sync(0xffffffffu, incl, off);
                            if (lane >= off) incl += v;
                        }
                        if (lane < min(n_kept, n - r)) a.group_start[(int64_t)m.h * (a.m_q + 1) + moff + lane] = m.start + incl - sz;
                        const int begin = __shfl_sync(0xffffffffu, incl - sz, row_of & 31);
                        if (tok >= 0) {   // the token's number in the original order: from the block's place in the scene, or through the reorder index
                            const Geometry bg = unpack_geometry(m.geom);
                            const int orig = DIRECT ? (bg.s0 + own_t) * a.layout.tokens_per_frame + a.layout.n_special + (bg.y0 + own_y) * a.layout.grid_w + bg.x0 + own_x
                                                    : __ldg(a.pi + m.start + tok);
                            a.group_member[(int64_t)m.h * a.n_tokens + m.start + begin + slot] = orig;
                        }
                    }
                }
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    rw[ks] = *reinterpret_cast<const uint2*>(rows_of + 16 * ks + 4 * tq);
                    w_fragment(af0[ks], rw[ks], row_pair(g), row_pair(g + 8));
                }
            }
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar0 + 8 * st, seq >> 1 & 1u, a.status, kDevTimeoutMatchLoad))) {
                failed = true;
                ahead = !SPLIT && (t < 2 || more);
                break;
            }
            if (r == 0) {   // nothing merges here: the rows leave as they are
                if (t == 0 && lane < n) {
                    if (!m.special()) a.rank_q[(int64_t)m.h * a.n_tokens + m.start + lane] = moff + lane;
                    if (a.group_start) {   // every token is a group of its own
                        a.group_start[(int64_t)m.h * (a.m_q + 1) + moff + lane] = m.start + lane;
                        a.group_member[(int64_t)m.h * a.n_tokens + m.start + lane] = __ldg(a.pi + m.start + lane);
                    }
                }
            } else {
                // x fragments of 16 channels: for k step ks (16 tokens) one ldmatrix.x4.trans gives b0, b1 of channel tile 2 np and b0, b1 of
                // channel tile 2 np + 1.  The merged rows take the same channels of the stage, so 16 channels at a time are in registers.
                const int n_mt = n_kept > 16 ? 2 : 1;
                const uint32_t from = blk + (lane & 15) * kRowBytes;
                const float i0 = g < n_kept ? rcnt[g] : 0.f, i1 = g + 8 < n_kept ? rcnt[g + 8] : 0.f;
                const int j = (lane & 7) + ((lane >> 4) << 3);   // row whose address this lane gives (matrices: rows 0-7 x two tiles, rows 8-15 x two)
#pragma unroll
                for (int np = 0; np < 4; ++np) {
                    uint32_t bf[2][4];
                    const uint32_t chunk = ((2 * np + (lane >> 4)) ^ (lane & 7)) << 4, to = blk + j * kRowBytes + (((2 * np + ((lane >> 3) & 1)) ^ (lane & 7)) << 4);
                    ldmatrix_x4_trans(bf[0], from + chunk);
                    if (n_ks > 1) ldmatrix_x4_trans(bf[1], from + 16 * kRowBytes + chunk);
                    __syncwarp();   // every lane has its fragments
                    auto rows_out = [&](const uint32_t (&w)[2][4], int mt, float i0, float i1) {
                        float p[2][4];
                        mma_first(p[0], w[0], bf[0][0], bf[0][1]);
                        mma_first(p[1], w[0], bf[0][2], bf[0][3]);
                        if (n_ks > 1) {
                            mma_bf16_16816(p[0], w[1], bf[1][0], bf[1][1]);
                            mma_bf16_16816(p[1], w[1], bf[1][2], bf[1][3]);
                        }
                        // rows past the last kept one become zeros (not 0 x something: the stage must stay finite)
                        const bool w0 = 16 * mt + g < n_kept, w1 = 16 * mt + g + 8 < n_kept;
                        stmatrix_x4(to + mt * 16 * kRowBytes, w0 ? pack2_bf16(p[0][0] * i0, p[0][1] * i0) : 0u,
                                    w0 ? pack2_bf16(p[1][0] * i0, p[1][1] * i0) : 0u, w1 ? pack2_bf16(p[0][2] * i1, p[0][3] * i1) : 0u,
                                    w1 ? pack2_bf16(p[1][2] * i1, p[1][3] * i1) : 0u);
                    };
                    rows_out(af0, 0, i0, i1);
                    if (n_mt == 2) {
                        uint32_t w[2][4];
                        w_fragment(w[0], rw[0], row_pair(g + 16), row_pair(g + 24));
                        w_fragment(w[1], rw[1], row_pair(g + 16), row_pair(g + 24));
                        rows_out(w, 1, g + 16 < n_kept ? rcnt[g + 16] : 0.f, g + 24 < n_kept ? rcnt[g + 24] : 0.f);
                    }
                }
                __syncwarp();
                n_out = min(n_kept, t == 0 && a.moff_q_var ? n : n - r);   // (a corrupt map cannot overrun; after outlier filtering more than n - r may be kept)
            }
            if (t == 0 && more) target_next[0] = load_target(meta_next, 0);   // (in flight during the stores and the next tensors)
            if (t == 1 && more) target_next[1] = load_target(meta_next, 1);
            if (DIRECT && r == 0 && !m.special()) {   // (the tokens of a clipped block are not consecutive rows)
                const Geometry bg = unpack_geometry(m.geom);
                for (int q = lane; q < n_out * 8; q += 32) {
                    const int row = row_of_token(box, bg, q >> 3);
                    out[q] = *reinterpret_cast<const uint4*>(rows + row * kRowBytes + (((q & 7) ^ (row & 7)) << 4));
                }
            } else {   // chunk c of row j sits at c ^ (j & 7); a lane's rows are 4 apart: two offsets serve all of them
                const int j0 = lane >> 3, ch = lane & 7;
                const unsigned char* even = rows + j0 * kRowBytes + ((ch ^ j0) << 4);
                const unsigned char* odds = rows + j0 * kRowBytes + ((ch ^ (j0 + 4)) << 4);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (4 * i >= n_out) break;   // (uniform)
                    if (4 * i + j0 < n_out) out[32 * i + lane] = *reinterpret_cast<const uint4*>(((i & 1) ? odds : even) + i * 4 * kRowBytes);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the merged rows were written by ordinary stores, the refill is not
            __syncwarp();
            if (!SPLIT && lane == 0) {   // the tensor after the next one takes this stage: V behind Q, then Q and K of the next unit
                if (t == 0)
                    issue(2, st, m);
                else if (more)
                    issue(t - 1, st, meta_next);
            }
        }
        if (failed) break;
    }
    if (failed)   // give copies that may still be in flight a bounded chance to land before the shared memory is released
        for (uint32_t i = seq; i <= seq + (ahead ? 1 : 0); ++i) mbar_wait_bounded(bar0 + 8 * (i & 1u), i >> 1 & 1u, a.status, kDevTimeoutMatchLoad);
}

int small_grid(int64_t units, int sm_count, int ctas_per_sm) {
    const int64_t grid = (units + kWarps - 1) / kWarps, cap = (int64_t)(sm_count < 1 ? 1 : sm_count) * ctas_per_sm;
    return (int)(grid > cap ? cap : (grid < 1 ? 1 : grid));
}

}  // namespace

namespace {
template <int TILES>
cudaError_t launch_match_tiles(const MatchArgs& a, int sm_count, cudaStream_t stream) {
    CUtensorMap mq, mk;
    const int64_t N = a.n_tokens;
    const bool direct = a.geom != nullptr;
    if (direct) {
        if (!encode_block_map(&mq, a.src[0], a.layout, a.heads) || !encode_block_map(&mk, a.src[1], a.layout, a.heads)) return cudaErrorInvalidValue;
    } else if (!encode_rows_tensor_map(&mq, a.xr[0], N, a.heads, kHeadDim, N * kHeadDim, 16 * TILES) ||
               !encode_rows_tensor_map(&mk, a.xr[1], N, a.heads, kHeadDim, N * kHeadDim, 16 * TILES)) {
        return cudaErrorInvalidValue;
    }
    const int64_t units = (int64_t)a.heads * a.n_blocks;
    auto launch = [&](auto kernel, int parts) {
        // Tasks of one tensor are dealt out evenly where there are few rounds of them, so that the last is no nearly empty one and the merge kernel's CTAs find room
        // earlier.  64-token blocks, ratio 0.8, calls with all warps / evenly dealt: 1.4 rounds 39.2 / 38.1 us, 2.7 65.1 / 64.6, 4.1 112.7 / 111.4, 5.4 166.2 / 166.6, 8.1
        // 172.1 / 173.0.
        const int64_t tasks = units * parts, warps = (int64_t)match_ctas(TILES) * kWarps * sm_count, rounds = (tasks + warps - 1) / warps;
        const int64_t dealt = parts == 2 && rounds > 1 && rounds <= 5 ? (tasks + rounds - 1) / rounds : tasks;
        return launch_kernel(kernel, small_grid(dealt, sm_count, match_ctas(TILES)), kWarps * 32, kMatchSmem, stream, mq, mk, a);
    };
    // With no more than one tensor per warp the tensors of a unit go to different warps: the call then waits for one, not two
    // (512 units: 11.3 -> 9.4 us, in the merge kernel below 13.1 -> 9.0).
    if (2 * units <= (int64_t)match_ctas(TILES) * kWarps * sm_count)
        return launch(direct ? match_small_kernel<TILES, true, false, true> : match_small_kernel<TILES, false, false, true>, 2);
    constexpr bool UNITS = TILES == 2;
    return launch(direct ? match_small_kernel<TILES, true, UNITS, false> : match_small_kernel<TILES, false, UNITS, false>, UNITS ? 1 : 2);
}
}  // namespace
cudaError_t launch_match_small(const MatchArgs& a, int max_block_tokens, int sm_count, cudaStream_t stream) {
    return max_block_tokens <= 32 ? launch_match_tiles<2>(a, sm_count, stream) : launch_match_tiles<4>(a, sm_count, stream);
}

cudaError_t launch_merge_small(const MergeArgs& a, int sm_count, cudaStream_t stream) {
    MergeMaps m;
    const bool direct = a.geom != nullptr;
    if (!encode_merge_maps(&m, a, 32)) return cudaErrorInvalidValue;
    const int sp_units = direct ? (a.layout.n_special > 0 ? a.layout.frames : 0) : (a.n_special_total + 31) / 32;
    const int64_t units = (int64_t)a.heads * (a.n_blocks + sp_units);
    auto launch = [&](auto kernel, int parts, int ctas) { return launch_kernel(kernel, small_grid(units * parts, sm_count, ctas), kWarps * 32, kMergeSmem, stream, m, a); };
    if (3 * units <= 2ll * kWarps * sm_count) return launch(direct ? merge_small_kernel<2, true, true> : merge_small_kernel<2, false, true>, 3, 2);
    if (unit_ctas(units, sm_count) == 3) return launch(direct ? merge_small_kernel<3, true, false> : merge_small_kernel<3, false, false>, 1, 3);   // 80 registers, else 111
    return launch(direct ? merge_small_kernel<2, true, false> : merge_small_kernel<2, false, false>, 1, 2);
}

cudaError_t configure_small_blocks() {
    cudaError_t e = cudaSuccess;
    auto set = [&](auto kernel, int bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    set(match_small_kernel<2, false, true, false>, kMatchSmem);
    set(match_small_kernel<2, true, true, false>, kMatchSmem);
    set(match_small_kernel<2, false, false, true>, kMatchSmem);
    set(match_small_kernel<2, true, false, true>, kMatchSmem);
    set(match_small_kernel<4, false, false, false>, kMatchSmem);
    set(match_small_kernel<4, true, false, false>, kMatchSmem);
    set(match_small_kernel<4, false, false, true>, kMatchSmem);
    set(match_small_kernel<4, true, false, true>, kMatchSmem);
    set(merge_small_kernel<2, false, false>, kMergeSmem);
    set(merge_small_kernel<2, false, true>, kMergeSmem);
    set(merge_small_kernel<2, true, false>, kMergeSmem);
    set(merge_small_kernel<2, true, true>, kMergeSmem);
    set(merge_small_kernel<3, false, false>, kMergeSmem);
    set(merge_small_kernel<3, true, false>, kMergeSmem);
    return e;
}

}  // namespace httm
