// Matching (65 .. 256 tokens) and merging (33 .. 256) of merging blocks (Eq. 1, Sec. 3.2).  A TEAM of W warps, a CTA of its own, works
// off a UNIT = one (head, block) with all its tensors; a thread owns P rows of the stage, so that a team takes blocks of
// 32 W P tokens: (W, P) = (1, 2), (4, 1) and (8, 1) for blocks of up to 64, 128 and 256 tokens.
// (Blocks of up to 64 tokens are matched by the small-block kernel.)
//
// What bounds them is instructions and their latency, not memory (2 - 3.3 of 6.5 TB/s).  With one warp per (tensor, head, block) and
// all of its tokens (16 / 12 / 6 warps per SM, as many blocks as shared memory takes) a 128-token block kept its warp busy for
// 17 us while 27 - 40 % of the issue slots were used.  A team of four shares that out; a second stage takes the next tensor's
// load, and table entries, geometry and map entries are fetched one unit ahead.  A block of up to 64 tokens stays with one
// warp: two of them spend as many instructions again on what every warp of a team does for itself.
// Measured, before / after (a call: back to back with others, so with what the kernels do to their neighbours):
//   128-token blocks, 32 976 tokens x 16 heads, ratio 0.9: match 79 / 44 us, merge 70 / 50 us, call 227 / 166 us; (2, 2): 47, 51, 168;
//   64-token blocks, 137 400 tokens, ratio 0.8: merge 200 / 180 us, (2, 1): 215;
//   48-token blocks, clipped, 7 898 tokens, ratio 0.6, with a team that matched them too: call 102 / 94 us; (2, 1): 106 us.
#include "httm_blocks.cuh"
#include "httm_launch.cuh"

namespace httm {

namespace {

__host__ __device__ constexpr int team_tokens(int w, int p) { return 32 * w * p; }   // largest block
template <int W>
__device__ __forceinline__ void team_sync() {
    if (W == 1) __syncwarp();
    else __syncthreads();
}
template <int W>
__device__ __forceinline__ bool team_any(bool x) {
    if (W > 1) return __syncthreads_or(x);
    const bool any = __any_sync(0xffffffffu, x);
    __syncwarp();
    return any;
}

// ------------------------------------------------------------------------------------ match
// Per tensor: squared norms of the team's rows (diagonals of a 16-row tile against itself), then the cosines of a warp's 32 rows
// with every dst token, 8 dst tokens at a time gathered by giving ldmatrix their row addresses (m16n8k16, exact bf16
// products, fp32 accumulation), best dst per row (ties: lowest).  The r src with the best scores merge (ties: lowest position
// first): the warps of the team look for the line between them and the others (choose).
struct MatchAux {   // shared memory behind the two stages
    int inv, keys, best, dst_row, dst_pos, src, bars, bytes;
};
__host__ __device__ constexpr MatchAux match_aux(int tokens) {
    MatchAux a{};
    a.inv = 0;                         // float [tokens] inverse norms of the stage's rows
    a.keys = a.inv + 4 * tokens;       // uint32 [tokens] order-preserving keys of the src tokens' scores, 0 for the others
    a.best = a.keys + 4 * tokens;      // int [tokens] best dst
    a.dst_row = a.best + 4 * tokens;   // int [tokens / 4] stage row of every dst token (the last one repeated)
    a.dst_pos = a.dst_row + tokens;    // int [tokens / 4] its number in the block
    a.src = a.dst_pos + tokens;        // uint8 [tokens] row holds a src token
    a.bars = a.src + tokens;
    a.bytes = a.bars + 16;
    return a;
}
struct MergeAux {
    int rows, cnt, kept, share, bars, bytes;
};
__host__ __device__ constexpr MergeAux merge_aux(int tokens) {
    MergeAux a{};
    a.rows = 0;                           // bf16 [unit parity][map][tokens] merged row of the token in a stage row (-1: none),
                                          // the tokens of a 16-row step in fragment order
    a.cnt = a.rows + 8 * tokens;          // int [unit parity][map][tokens] members of a merged row
    a.kept = a.cnt + 16 * tokens;         // uint32 [map][8] kept tokens by stage row
    a.share = a.kept + 2 * 4 * 8;         // float [tokens + 1] 1 / c
    a.bars = a.share + 4 * tokens + 16;
    a.bytes = a.bars + 16;
    return a;
}
// Match and merge teams of a size ask for the same shared memory.  The merge CTAs move in one by one as match CTAs of the kernel before end
// (launch ahead of the predecessor's end), and a hole of another size than theirs stays partly unused: with 19 408 and 20 320
// bytes a third of the merge CTAs found no place until others had finished (137 344 tokens, 64-token blocks, when a team matched those: 100 us).
// Teams of one warp now follow the small-block kernel's match CTAs of 66 688 bytes, and how large these are counts too: asking for 73 984 a call on 32 976 tokens in 64-token
// blocks, ratio 0.8, takes 312 us instead of 297.  For blocks of at most 32 tokens it does not: match and merge with 73 984 bytes each, the deviation kernel's, instead of 66 688 and
// 69 248 make no difference of more than 0.2 % in calls on 1 044 .. 65 952 tokens, with outlier filtering or without.
constexpr int team_smem(int w, int p) {
    return 2 * team_tokens(w, p) * kRowBytes + merge_aux(team_tokens(w, p)).bytes + 1024 /*alignment slack*/;
}
static_assert(match_aux(128).bytes <= merge_aux(128).bytes && match_aux(256).bytes <= merge_aux(256).bytes, "a match team fits in what the merge team needs");
constexpr int team_ctas(int w, int p) {   // CTAs per SM: all of a persistent grid have to be resident
    const int by_warps = (p == 1 ? 24 : 12) / w, by_smem = 228 * 1024 / (team_smem(w, p) + 1024);
    return by_warps < by_smem ? by_warps : by_smem;
}

// Is this thread's key (row 32 warp + lane, 0: no src token) one of the r largest of n_rows stage rows, equal ones at the lowest rows first?  (Fewer than all merge.)
// Every warp of the team looks for a value with r keys above it, by bisection between the smallest and the largest key: with distinct keys about as many steps as the
// logarithm of their number, 32 at most.  Every thread counting the keys that come before its own took a warp of a 128-token block 400 instructions, this 150: 32 976 tokens x 16 heads,
// ratio 0.6 a call 1021 -> 980 us, 0.7 655 -> 615; 52 318 tokens x 8 heads, ratios 0.56 and 0.74, match 87 -> 57 us.
template <int NK>
__device__ __forceinline__ bool choose(const uint32_t* keys, int n_rows, int r, uint32_t mine, int warp, int lane) {
    uint32_t k[NK], hi = 0u, lo = 0xffffffffu;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
        k[j] = 32 * j + lane < n_rows ? keys[32 * j + lane] : 0u;
        hi = max(hi, k[j]);
        lo = min(lo, k[j] - 1u);   // (0 becomes the largest)
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);   // at most r keys above hi, at least r above lo
    int above = 0;                             // keys above hi
#pragma unroll 1
    while (hi - lo > 1u) {
        const uint32_t bar = lo + (hi - lo) / 2;
        int c = 0;
#pragma unroll
        for (int j = 0; j < NK; ++j) c += k[j] > bar ? 1 : 0;
        c = __reduce_add_sync(0xffffffffu, c);
        if (c > r) {
            lo = bar;
        } else {
            hi = bar;
            above = c;
            if (c == r) break;
        }
    }
    if (above == r) return mine > hi;
    // more keys equal to hi than are wanted of them: those at the lowest rows
    int before = 0;
#pragma unroll
    for (int j = 0; j < NK; ++j) {
        const unsigned equal = __ballot_sync(0xffffffffu, k[j] == hi);
        before += j < warp ? __popc(equal) : (j == warp ? __popc(equal & ((1u << lane) - 1u)) : 0);
    }
    return mine > hi || (mine == hi && before < r - above);
}

template <int W, bool DIRECT>
__global__ void __launch_bounds__(32 * W, team_ctas(W, 1))
match_team_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ MatchArgs a) {
    static_assert(W > 1, "a team has several warps, a thread one token");
    constexpr int NMAX = team_tokens(W, 1), MT = 2, MAX_DST = NMAX / 4;   // MT: 16-row tiles per warp
    constexpr uint32_t STAGE = NMAX * kRowBytes;
    constexpr MatchAux X = match_aux(NMAX);
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + align_pad(smem_raw);
    unsigned char* aux = smem + 2 * STAGE;
    float* inv = reinterpret_cast<float*>(aux + X.inv);
    uint32_t* keys = reinterpret_cast<uint32_t*>(aux + X.keys);
    int* best = reinterpret_cast<int*>(aux + X.best);
    int* dst_row = reinterpret_cast<int*>(aux + X.dst_row);
    int* dst_pos = reinterpret_cast<int*>(aux + X.dst_pos);
    unsigned char* src = aux + X.src;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, tq = lane & 3, odd = tq & 1;   // accumulator layout: rows g, g + 8; columns 2 tq, 2 tq + 1
    const uint32_t stage0 = smem_u32(smem), bar0 = smem_u32(aux + X.bars);
    if (tid == 0) {
        mbar_init(bar0, 1);
        mbar_init(bar0 + 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    team_sync<W>();

    Box box{};
    if (DIRECT) box.set(a.layout);
    const int64_t n_units = (int64_t)a.heads * a.n_blocks;
    UnitCursor next;
    next.init(blockIdx.x, gridDim.x, a.n_blocks);
    auto issue = [&](int t, const int4& geom, int start, int h) {   // thread 0 only
        const uint32_t mb = bar0 + 8 * t;
        const CUtensorMap* m = t == 0 ? &map_q : &map_k;
        if (DIRECT) {
            const Geometry bg = unpack_geometry(geom);
            mbar_expect_tx(mb, (uint32_t)box.rows * kRowBytes);
            tma_block_load(stage0 + t * STAGE, m, mb, bg.x0, bg.y0, bg.s0, h);
        } else {
            mbar_expect_tx(mb, STAGE);
            tma_rows_load(stage0 + t * STAGE, m, mb, start, h);
        }
    };
    BlockInfo bi_next{};
    int4 geom_next{};
    int h_next = 0;
    auto fetch = [&]() {
        bi_next = a.blocks[next.u];
        if (DIRECT) geom_next = load_geometry(a.geom, next.u);
        h_next = next.h;
    };
    if (blockIdx.x < n_units) fetch();
    depend_wait();
    dependents_launch();
    clear_words(a.clear, blockIdx.x, gridDim.x);
    if (blockIdx.x < n_units && tid == 0) {
        issue(0, geom_next, bi_next.start, h_next);
        issue(1, geom_next, bi_next.start, h_next);
    }
    // ldmatrix offsets of a 16-row tile: rows 0-7 / 8-15 (lane bit 3), k chunk 2 ks / 2 ks + 1 (lane bit 4); chunk c of row j sits at c ^ (j & 7)
    uint32_t a_off[4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) a_off[ks] = (warp * 32 + (lane & 15)) * kRowBytes + (((2 * ks + (lane >> 4)) ^ (lane & 7)) << 4);
    int shape_a = -1, shape_b = -1;   // shape of the blocks at hand: the tables and tok are made for it
    int tok = -1;                     // token in this thread's stage row
    const int row0 = warp * 32, own = row0 + lane;
    int it = 0;
    int failed = -1;   // tensor whose load did not arrive
    for (int64_t unit = blockIdx.x; unit < n_units; unit += gridDim.x, ++it) {
        const BlockInfo bi = bi_next;
        const int4 geom = geom_next;
        const int h = h_next, n = bi.n;
        const bool more = unit + gridDim.x < n_units;
        if (more) {
            next.advance();
            fetch();   // in flight while this unit is worked off
        }
#pragma unroll 1
        for (int t = 0; t < 2; ++t) {
            const int r = t == 0 ? bi.r_q : bi.r_k, nd = t == 0 ? bi.nd_q : bi.nd_k;
            int32_t* A = a.assign[t] + (int64_t)h * a.n_tokens + bi.start;
            const bool arrived = mbar_wait_bounded(bar0 + 8 * t, it & 1, a.status, kDevTimeoutMatchLoad);
            if (r == 0 || nd > MAX_DST) {   // nothing merges, or an anchored block with more dst tokens (match_anchor_kernel)
                if (team_any<W>(!arrived)) {
                    failed = t;
                    break;
                }
                if (r == 0)
                    for (int j = tid; j < n; j += 32 * W) A[j] = bi.start + j;
                if (more && tid == 0) issue(t, geom_next, bi_next.start, h_next);
                continue;
            }
            const int n_rows = DIRECT ? box.rows : n;   // rows of the stage that may hold tokens
            {
                const int sa = n | (nd << 10) | (bi.n_rule << 20), sb = DIRECT ? shape_key(geom) : 0;
                if (sa != shape_a || sb != shape_b) {   // (uniform)
                    team_sync<W>();   // the tables may still be read for the previous tensor
                    shape_a = sa;
                    shape_b = sb;
                    const int n_rule = bi.n_rule;   // n (evenly spaced dst tokens) or n_dst (the first n_dst tokens: first-frame anchoring)
                    const Geometry bg = unpack_geometry(geom);
                    if (tid < MAX_DST) {
                        const int pos = small_div((min(tid, nd - 1) + 1) * n_rule + nd - 1, nd) - 1;
                        dst_pos[tid] = pos;
                        dst_row[tid] = DIRECT ? row_of_token(box, bg, pos) : pos;
                    }
                    tok = DIRECT ? token_of_row(box, bg, own) : (own < n ? own : -1);
                    src[own] = tok >= 0 && !(tok < n_rule && small_div((tok + 1) * nd, n_rule) > small_div(tok * nd, n_rule)) ? 1 : 0;
                }
            }
            const uint32_t blk = stage0 + t * STAGE;
            // ---- the warp's rows and their inverse norms
            uint32_t af[MT][4][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                if (row0 + mt * 16 < n_rows) {   // warp-uniform
                    float lo[4], hi[4];
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        uint32_t* f = af[mt][ks];
                        ldmatrix_x4(f, blk + mt * 16 * kRowBytes + a_off[ks]);
                        if (ks == 0) {
                            mma_first(lo, f, f[0], f[2]);   // against rows 0-7 of the tile
                            mma_first(hi, f, f[1], f[3]);   // against rows 8-15
                        } else {
                            mma_bf16_16816(lo, f, f[0], f[2]);
                            mma_bf16_16816(hi, f, f[1], f[3]);
                        }
                    }
                    if (tq == (g >> 1)) {   // this lane holds the diagonal entries of rows g and g + 8
                        inv[row0 + mt * 16 + g] = inv_norm((g & 1) ? lo[1] : lo[0]);
                        inv[row0 + mt * 16 + 8 + g] = inv_norm((g & 1) ? hi[3] : hi[2]);
                    }
                }
            }
            if (team_any<W>(!arrived)) {   // inverse norms and tables visible
                failed = t;
                break;
            }
            // ---- best dst of every row
            if (row0 < n_rows) {
                float top[MT][2];   // [tile][rows g, g + 8]
                int arg[MT][2];
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    top[mt][0] = top[mt][1] = -INFINITY;
                    arg[mt][0] = arg[mt][1] = 0;
                }
                const int n_tiles = min(MT, (n_rows - row0 + 15) >> 4);
#pragma unroll 1
                for (int d0 = 0; d0 < nd; d0 += 8) {   // (places past the last dst token repeat it: they never beat it)
                    const int row = dst_row[d0 + (lane & 7)];
                    const float w = inv[row];
                    uint32_t bf[4][2];
#pragma unroll
                    for (int kp = 0; kp < 2; ++kp) {   // one ldmatrix.x4 = k steps 2 kp and 2 kp + 1
                        uint32_t rr[4];
                        ldmatrix_x4(rr, blk + row * kRowBytes + (((4 * kp + (lane >> 3)) ^ (row & 7)) << 4));
                        bf[2 * kp][0] = rr[0];
                        bf[2 * kp][1] = rr[1];
                        bf[2 * kp + 1][0] = rr[2];
                        bf[2 * kp + 1][1] = rr[3];
                    }
                    const float w0 = __shfl_sync(0xffffffffu, w, 2 * tq), w1 = __shfl_sync(0xffffffffu, w, 2 * tq + 1);
                    const int da = d0 + 2 * tq;
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        if (mt < n_tiles) {
                            float c[4];
                            mma_first(c, af[mt][0], bf[0][0], bf[0][1]);
#pragma unroll
                            for (int ks = 1; ks < 4; ++ks) mma_bf16_16816(c, af[mt][ks], bf[ks][0], bf[ks][1]);
#pragma unroll
                            for (int hrow = 0; hrow < 2; ++hrow) {
                                const float s0 = c[2 * hrow] * w0, s1 = c[2 * hrow + 1] * w1, m = fmaxf(s0, s1);
                                if (m > top[mt][hrow]) {
                                    top[mt][hrow] = m;
                                    arg[mt][hrow] = da + (s0 != m ? 1 : 0);   // (also where s0 is not a number)
                                }
                            }
                        }
                    }
                }
                // lanes 0, 1 of a row's four split the rows g and g + 8, then meet lanes 2, 3 (ties: lowest dst)
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    if (mt < n_tiles) {
                        float tp = odd ? top[mt][1] : top[mt][0];
                        int ag = odd ? arg[mt][1] : arg[mt][0];
                        const float sv = odd ? top[mt][0] : top[mt][1];
                        const int sg = odd ? arg[mt][0] : arg[mt][1];
#pragma unroll
                        for (int off = 1; off <= 2; off <<= 1) {
                            const float ov = __shfl_xor_sync(0xffffffffu, off == 1 ? sv : tp, off);
                            const int oa = __shfl_xor_sync(0xffffffffu, off == 1 ? sg : ag, off);
                            if (ov > tp || (ov == tp && oa < ag)) {
                                tp = ov;
                                ag = oa;
                            }
                        }
                        if (tq < 2) {
                            const int rho = row0 + mt * 16 + odd * 8 + g;
                            keys[rho] = src[rho] ? score_key(tp * inv[rho]) : 0u;
                            best[rho] = ag;
                        }
                    }
                }
            }
            team_sync<W>();   // keys visible; every warp has read the stage
            if (more && tid == 0) issue(t, geom_next, bi_next.start, h_next);
            // ---- the r src with the best scores merge (ties: lowest position first; rows are in token order)
            const int n_out = n - nd - r;
            const uint32_t key = tok >= 0 ? keys[own] : 0u;   // (0: not a src token)
            bool merged = key != 0;
            if (n_out > 0) merged = choose<NMAX / 32>(keys, (n_rows + 15) & ~15, r, key, warp, lane);
            if (tok >= 0) A[tok] = bi.start + (merged ? dst_pos[best[own]] : tok);
        }
        if (failed >= 0) break;
    }
    if (failed >= 0) {   // give copies that may still be in flight a bounded chance to land before the shared memory is released
        mbar_wait_bounded(bar0, (it + failed) & 1, a.status, kDevTimeoutMatchLoad);   // (past Q: its next load has been issued)
        mbar_wait_bounded(bar0 + 8, it & 1, a.status, kDevTimeoutMatchLoad);
    }
}

// ------------------------------------------------------------------------------------ merge
// The contraction of httm_small_blocks.cu, merged_sum = W x, for a team: one thread per stage row makes the groups, then every
// warp takes 64 / W channels (W = 8: 16 channels and every other tile) of all tiles of 16 merged rows, tokens in steps of 16,
// skipping steps without a member of the tile's rows.  K's groups serve V.  Tensor i of the CTA's sequence Q K V Q K V .. lies
// in stage i & 1.  The next unit's groups are made between the tensors of this one (who is kept beside K, merged rows and
// counts beside V), so that the barrier behind each tensor is the only one.
template <int W, int P, bool DIRECT>
__global__ void __launch_bounds__(32 * W, team_ctas(W, P)) merge_team_kernel(const __grid_constant__ MergeMaps maps, const __grid_constant__ MergeArgs a) {
    constexpr int NMAX = team_tokens(W, P), T = 32 * W;
    constexpr uint32_t STAGE = NMAX * kRowBytes;
    constexpr MergeAux X = merge_aux(NMAX);
    static_assert(W == 1 || W == 4 || W == 8, "how the channels are dealt to the warps");
    constexpr int NP = W == 1 ? 4 : 1;   // pairs of 8-channel tiles per warp
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + align_pad(smem_raw);
    unsigned char* aux = smem + 2 * STAGE;
    __nv_bfloat16* rows = reinterpret_cast<__nv_bfloat16*>(aux + X.rows);
    int* cnt = reinterpret_cast<int*>(aux + X.cnt);
    uint32_t* kept = reinterpret_cast<uint32_t*>(aux + X.kept);
    float* share = reinterpret_cast<float*>(aux + X.share);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, tq = lane & 3;   // accumulator layout: rows g, g + 8; columns 2 tq, 2 tq + 1
    const uint32_t stage0 = smem_u32(smem), bar0 = smem_u32(aux + X.bars);
    if (tid == 0) {
        mbar_init(bar0, 1);
        mbar_init(bar0 + 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < NMAX; i += T) share[i + 1] = 1.0f / (float)(i + 1);
    Box box{};
    if (DIRECT) {
        box.set(a.layout);
        for (int q = box.rows * 8 + tid; q < NMAX * 8; q += T) {   // rows that no block load writes enter the MMAs with weight 0: keep them finite
            *reinterpret_cast<uint4*>(smem + q * 16) = make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4*>(smem + STAGE + q * 16) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    team_sync<W>();
    const int own = warp * 32 * P + lane;   // this thread's stage rows: own + 32 p

    // units 0 .. n_blocks - 1 of a head are merging blocks, the rest special tokens (never merged: copied)
    const int sp_units = DIRECT ? (a.layout.n_special > 0 ? a.layout.frames : 0) : (a.n_special_total + 31) / 32;
    const int per_head = a.n_blocks + sp_units;
    const int64_t n_units = (int64_t)a.heads * per_head;
    struct Meta {
        int h, start, n, r_q, r_k, moff_q, moff_k;
        int4 geom;   // (of special tokens: .w = their frame + 1)
        __device__ bool special() const { return geom.w != 0; }
    };
    UnitCursor next;
    next.init(blockIdx.x, gridDim.x, per_head);
    auto fetch = [&]() {
        Meta m{};
        m.h = next.h;
        if (next.u >= a.n_blocks) {
            const int frame = next.u - a.n_blocks;
            m.start = m.moff_q = m.moff_k = frame * (DIRECT ? a.layout.n_special : 32);
            m.n = DIRECT ? a.layout.n_special : min(32, a.n_special_total - m.start);
            m.geom.w = frame + 1;
        } else {
            if (DIRECT) m.geom = load_geometry(a.geom, next.u);
            m.geom.w = 0;
            const BlockInfo bi = a.blocks[next.u];
            m.start = bi.start;
            m.n = bi.n;
            m.r_q = bi.r_q;
            m.r_k = bi.r_k;
            m.moff_q = bi.moff_q;
            m.moff_k = bi.moff_k;
        }
        return m;
    };
    auto issue = [&](int t, uint32_t st, const Meta& m) {   // thread 0 only
        const uint32_t mb = bar0 + 8 * st, dst = stage0 + st * STAGE;
        if (!DIRECT) {
            mbar_expect_tx(mb, STAGE);   // (rows past the head's end are zero filled)
            tma_rows_load(dst, &maps.block[t], mb, m.start, m.h);
        } else if (m.special()) {
            mbar_expect_tx(mb, (uint32_t)m.n * kRowBytes);
            asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
                         "l"(reinterpret_cast<uint64_t>(&maps.special[t])), "r"(mb), "r"(0), "r"(0), "r"(m.geom.w - 1), "r"(m.h)
                         : "memory");
        } else {
            const Geometry bg = unpack_geometry(m.geom);
            mbar_expect_tx(mb, (uint32_t)box.rows * kRowBytes);
            tma_block_load(dst, &maps.block[t], mb, bg.x0, bg.y0, bg.s0, m.h);
        }
    };
    // the tokens in this thread's stage rows (numbers in the block, -1: none) and the tokens these are merged into
    struct Targets {
        int tok[P], to[2][P];
    };
    auto load_targets = [&](const Meta& m) {
        Targets x;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int rho = own + 32 * p;
            x.tok[p] = !DIRECT || m.special() ? (rho < m.n ? rho : -1) : token_of_row(box, unpack_geometry(m.geom), rho);
            x.to[0][p] = x.to[1][p] = -1;
            const int64_t at = (int64_t)m.h * a.n_tokens + m.start + x.tok[p];
            if (x.tok[p] >= 0 && m.r_q > 0) x.to[0][p] = ld_global(a.assign[0] + at) - m.start;
            if (x.tok[p] >= 0 && m.r_k > 0) x.to[1][p] = ld_global(a.assign[1] + at) - m.start;
        }
        return x;
    };
    // groups of a unit, first half: the stage row of the token each token is merged into; kept tokens; counts to zero
    auto find_kept = [&](const Meta& m, Targets& x, int par) {
#pragma unroll
        for (int map = 0; map < 2; ++map)
#pragma unroll
            for (int p = 0; p < P; ++p) {
                int rep = -1;
                if (x.tok[p] >= 0 && (map == 0 ? m.r_q : m.r_k) > 0) {
                    rep = x.to[map][p];
                    if (rep < 0 || rep >= m.n) {   // corrupt map: record, treat as kept
                        atomicCAS(a.status, kDevOk, kDevBadIndex);
                        rep = x.tok[p];
                    }
                    if (DIRECT) rep = row_of_token(box, unpack_geometry(m.geom), rep);
                }
                x.to[map][p] = rep;
                const unsigned mask = __ballot_sync(0xffffffffu, rep == own + 32 * p);
                if (lane == 0) kept[map * 8 + warp * P + p] = mask;
                cnt[(2 * par + map) * NMAX + own + 32 * p] = 0;
            }
    };
    // second half (a barrier later): merged row of every token = rank of its representative among the kept tokens
    auto rank_kept = [&](const Meta& m, const Targets& x, int par, int* n_kept) {
        const int at = fragment_order(own);
#pragma unroll
        for (int map = 0; map < 2; ++map) {
            int row[P], total = 0;
#pragma unroll
            for (int p = 0; p < P; ++p) row[p] = 0;
#pragma unroll
            for (int w = 0; w < W * P; ++w) {
                const uint32_t mask = kept[map * 8 + w];
                const int c = __popc(mask);
                total += c;
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const int rep = x.to[map][p];
                    if (w < (rep >> 5)) row[p] += c;
                    if (w == (rep >> 5)) row[p] += __popc(mask & ((1u << (rep & 31)) - 1u));
                }
            }
            n_kept[map] = total;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                if (x.to[map][p] >= 0)
                    atomicAdd(&cnt[(2 * par + map) * NMAX + row[p]], 1);
                else
                    row[p] = -1;
                rows[(2 * par + map) * NMAX + at + 32 * p] = __float2bfloat16_rn((float)row[p]);
                if (map == 0 && x.tok[p] >= 0 && !m.special()) a.rank_q[(int64_t)m.h * a.n_tokens + m.start + x.tok[p]] = m.moff_q + (m.r_q > 0 ? row[p] : x.tok[p]);
            }
        }
    };
    Meta m{}, meta_next{};
    if (blockIdx.x < n_units) m = fetch();
    auto issue_first = [&]() {
        if (blockIdx.x < n_units && tid == 0) {
            issue(0, 0, m);
            issue(1, 1, m);
        }
    };
    if (a.early) issue_first();
    depend_wait();
    dependents_launch();
    if (!a.early) issue_first();
    int n_kept[2] = {0, 0};
    if (blockIdx.x < n_units) {
        Targets x = load_targets(m);
        find_kept(m, x, 0);
        team_sync<W>();
        rank_kept(m, x, 0, n_kept);
        team_sync<W>();
    }
    uint32_t seq = 0;   // tensors so far
    int par = 0;
    bool failed = false;
    for (int64_t unit = blockIdx.x; unit < n_units; unit += gridDim.x, par ^= 1) {
        const bool more = unit + gridDim.x < n_units;
        Targets x{};
        int kept_next[2] = {0, 0};
        if (more) {   // in flight beside Q
            next.advance();
            meta_next = fetch();
            x = load_targets(meta_next);
        }
        const int n_ks = ((DIRECT ? box.rows : m.n) + 15) >> 4;   // 16-row steps of the stage that may hold tokens
#pragma unroll 1
        for (int t = 0; t < 3; ++t, ++seq) {
            const uint32_t st = seq & 1u;
            const int r = t == 0 ? m.r_q : m.r_k, moff = t == 0 ? m.moff_q : m.moff_k, m_len = t == 0 ? a.m_q : a.m_k;
            __nv_bfloat16* out = a.merged[t] + ((int64_t)m.h * m_len + moff) * kHeadDim;
            const bool arrived = mbar_wait_bounded(bar0 + 8 * st, (seq >> 1) & 1u, a.status, kDevTimeoutMatchLoad);
            const uint32_t blk = stage0 + st * STAGE;
            if (r == 0) {   // nothing merges here: the rows leave as they are (chunk c of row j sits at c ^ (j & 7))
                const unsigned char* stage = smem + st * STAGE;
                const Geometry bg = unpack_geometry(m.geom);
                if (arrived)
                    for (int q = tid; q < m.n * 8; q += T) {
                        const int row = DIRECT && !m.special() ? row_of_token(box, bg, q >> 3) : q >> 3;
                        reinterpret_cast<uint4*>(out)[q] = *reinterpret_cast<const uint4*>(stage + row * kRowBytes + (((q & 7) ^ (row & 7)) << 4));
                    }
            } else {
                const int map = t == 0 ? 0 : 1;
                const __nv_bfloat16* row_of = rows + (2 * par + map) * NMAX;
                const int* members = cnt + (2 * par + map) * NMAX;
                const int k = t == 0 ? n_kept[0] : n_kept[1];
                const int n_mt = (k + 15) >> 4, n_out = min(k, m.n - r);   // (a corrupt map cannot overrun)
                const int np0 = W == 1 ? 0 : (warp & 3);
#pragma unroll 1
                for (int mt = W == 8 ? warp >> 2 : 0; mt < n_mt; mt += W == 8 ? 2 : 1) {
                    const int r0 = 16 * mt + g, r1 = r0 + 8;   // this lane's two accumulator rows
                    const uint32_t b0 = row_pair(r0), b1 = row_pair(r1);
                    float c[NP][2][4];
#pragma unroll
                    for (int i = 0; i < NP; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e) c[i][0][e] = c[i][1][e] = 0.f;
#pragma unroll 2
                    for (int ks = 0; ks < n_ks; ++ks) {
                        const uint2 rw = *reinterpret_cast<const uint2*>(row_of + 16 * ks + 4 * tq);
                        uint32_t af[4];
                        w_fragment(af, rw, b0, b1);
                        if (!__any_sync(0xffffffffu, (af[0] | af[1] | af[2] | af[3]) != 0u)) continue;   // no token of this step belongs to this tile
                        const int j = 16 * ks + (lane & 15);
#pragma unroll
                        for (int i = 0; i < NP; ++i) {
                            uint32_t bf[4];
                            ldmatrix_x4_trans(bf, blk + j * kRowBytes + (((2 * (np0 + i) + (lane >> 4)) ^ (j & 7)) << 4));
                            mma_bf16_16816(c[i][0], af, bf[0], bf[1]);
                            mma_bf16_16816(c[i][1], af, bf[2], bf[3]);
                        }
                    }
                    // a pair of lanes swaps words so that the even one stores two of the first tile, the odd one two of the second:
                    // whole 32-byte sectors of a row per store
                    const bool w0 = r0 < n_out, w1 = r1 < n_out;
                    const float i0 = w0 ? share[members[r0]] : 0.f, i1 = w1 ? share[members[r1]] : 0.f;
                    const bool odd = tq & 1;
#pragma unroll
                    for (int i = 0; i < NP; ++i)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float inv = e ? i1 : i0;
                            const uint32_t first = pack2_bf16(c[i][0][2 * e] * inv, c[i][0][2 * e + 1] * inv), second = pack2_bf16(c[i][1][2 * e] * inv, c[i][1][2 * e + 1] * inv);
                            const uint32_t other = __shfl_xor_sync(0xffffffffu, odd ? first : second, 1);
                            const uint2 v = odd ? make_uint2(other, second) : make_uint2(first, other);
                            const int at = (e ? r1 : r0) * 32 + (2 * (np0 + i) + (odd ? 1 : 0)) * 4 + (tq & 2);   // 32 words per row
                            if ((e ? w1 : w0) && arrived) *reinterpret_cast<uint2*>(reinterpret_cast<uint32_t*>(out) + at) = v;
                        }
                }
            }
            if (more && t == 1) find_kept(meta_next, x, par ^ 1);
            if (more && t == 2) rank_kept(meta_next, x, par ^ 1, kept_next);
            if (team_any<W>(!arrived)) {   // every warp is done with the stage and the tables
                failed = true;
                break;
            }
            if (tid == 0) {   // the tensor after the next one, into this stage
                if (t == 0)
                    issue(2, st, m);
                else if (more)
                    issue(t - 1, st, meta_next);
            }
        }
        if (failed) break;
        m = meta_next;
        n_kept[0] = kept_next[0];
        n_kept[1] = kept_next[1];
    }
    if (failed) {
        mbar_wait_bounded(bar0 + 8 * (seq & 1u), (seq >> 1) & 1u, a.status, kDevTimeoutMatchLoad);
        mbar_wait_bounded(bar0 + 8 * ((seq + 1) & 1u), ((seq + 1) >> 1) & 1u, a.status, kDevTimeoutMatchLoad);
    }
}

int team_grid(int64_t units, int sm_count, int ctas) {
    const int64_t cap = (int64_t)(sm_count < 1 ? 1 : sm_count) * ctas;
    return (int)(units > cap ? cap : (units < 1 ? 1 : units));
}

template <int W>
cudaError_t launch_match_t(const MatchArgs& a, int sm_count, cudaStream_t stream) {
    CUtensorMap mq, mk;
    const int64_t N = a.n_tokens;
    const bool direct = a.geom != nullptr;
    if (direct) {
        if (!encode_block_map(&mq, a.src[0], a.layout, a.heads) || !encode_block_map(&mk, a.src[1], a.layout, a.heads)) return cudaErrorInvalidValue;
    } else if (!encode_rows_tensor_map(&mq, a.xr[0], N, a.heads, kHeadDim, N * kHeadDim, team_tokens(W, 1)) ||
               !encode_rows_tensor_map(&mk, a.xr[1], N, a.heads, kHeadDim, N * kHeadDim, team_tokens(W, 1))) {
        return cudaErrorInvalidValue;
    }
    auto kernel = direct ? match_team_kernel<W, true> : match_team_kernel<W, false>;
    return launch_kernel(kernel, team_grid((int64_t)a.heads * a.n_blocks, sm_count, team_ctas(W, 1)), 32 * W, team_smem(W, 1), stream, mq, mk, a);
}
template <int W, int P>
cudaError_t launch_merge_t(const MergeArgs& a, int sm_count, cudaStream_t stream) {
    MergeMaps m;
    const bool direct = a.geom != nullptr;
    if (!encode_merge_maps(&m, a, team_tokens(W, P))) return cudaErrorInvalidValue;
    const int sp_units = direct ? (a.layout.n_special > 0 ? a.layout.frames : 0) : (a.n_special_total + 31) / 32;
    auto kernel = direct ? merge_team_kernel<W, P, true> : merge_team_kernel<W, P, false>;
    return launch_kernel(kernel, team_grid((int64_t)a.heads * (a.n_blocks + sp_units), sm_count, team_ctas(W, P)), 32 * W, team_smem(W, P), stream, m, a);
}

template <int W, int P>
cudaError_t configure_t() {
    cudaError_t e = cudaSuccess;
    auto set = [&](auto kernel, int bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    if constexpr (W > 1) {
        set(match_team_kernel<W, false>, team_smem(W, 1));
        set(match_team_kernel<W, true>, team_smem(W, 1));
    }
    set(merge_team_kernel<W, P, false>, team_smem(W, P));
    set(merge_team_kernel<W, P, true>, team_smem(W, P));
    return e;
}

}  // namespace

cudaError_t launch_match_mid(const MatchArgs& a, int max_block_tokens, int sm_count, cudaStream_t stream) {
    if (max_block_tokens <= 128) return launch_match_t<4>(a, sm_count, stream);
    return launch_match_t<8>(a, sm_count, stream);
}
cudaError_t launch_merge_mid(const MergeArgs& a, int max_block_tokens, int sm_count, cudaStream_t stream) {
    if (max_block_tokens <= 64) return launch_merge_t<1, 2>(a, sm_count, stream);
    if (max_block_tokens <= 128) return launch_merge_t<4, 1>(a, sm_count, stream);
    return launch_merge_t<8, 1>(a, sm_count, stream);
}
cudaError_t configure_mid_blocks() {
    cudaError_t e = configure_t<1, 2>();
    if (e == cudaSuccess) e = configure_t<4, 1>();
    if (e == cudaSuccess) e = configure_t<8, 1>();
    return e;
}

}  // namespace httm
