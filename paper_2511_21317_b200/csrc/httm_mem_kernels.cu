// HBM-bound kernels of the HTTM path: temporal reorder (gather), matching of first-frame blocks, outlier filtering, unmerge +
// inverse reorder, and the choice of the matching and merging kernels by block size.  sm_100a only.
#include "httm_internal.h"
#include "httm_launch.cuh"
#include "httm_blocks.cuh"

namespace httm {

// ------------------------------------------------------------------------------------
// a1. Temporal reorder (Sec. 3.3; Algorithm 1 "Reorder"): xr[h][p'] = x[h][pi[p']]
//     One 16-byte chunk per thread, 8 threads per token row, 4 rows in flight per thread.
// ------------------------------------------------------------------------------------
constexpr int kReorderThreads = 256;
constexpr int kReorderUnroll = 4;
constexpr int kReorderTokensPerCta = (kReorderThreads / 8) * kReorderUnroll;

template <bool NORMS>   // NORMS: also write 1 / max(|x|, 1e-12) of every Q and K token (the large-block matcher needs them)
__global__ void __launch_bounds__(kReorderThreads) reorder_kernel(const __grid_constant__ ReorderArgs a) {
    const int t = blockIdx.z, h = blockIdx.y;
    const int chunk = threadIdx.x & 7, slot = threadIdx.x >> 3;
    const int base = blockIdx.x * kReorderTokensPerCta;
    const __nv_bfloat16* src = a.src[t].ptr + (int64_t)h * a.src[t].stride_head + chunk * 8;
    const int64_t st = a.src[t].stride_token;
    __nv_bfloat16* dst = a.dst[t] + (int64_t)h * a.n_tokens * kHeadDim + chunk * 8;
    uint4 v[kReorderUnroll];
    int row[kReorderUnroll];
#pragma unroll
    for (int u = 0; u < kReorderUnroll; ++u) {
        const int p = base + u * (kReorderThreads / 8) + slot;
        row[u] = p < a.n_tokens ? __ldg(a.pi + p) : 0;
    }
    depend_wait();
    dependents_launch();
    if (t == 0 && h == 0) clear_words(a.clear, blockIdx.x, gridDim.x);
#pragma unroll
    for (int u = 0; u < kReorderUnroll; ++u) {
        const int p = base + u * (kReorderThreads / 8) + slot;
        v[u] = make_uint4(0u, 0u, 0u, 0u);
        if (p < a.n_tokens) v[u] = ld_global(reinterpret_cast<const uint4*>(src + (int64_t)row[u] * st));
    }
#pragma unroll
    for (int u = 0; u < kReorderUnroll; ++u) {
        const int p = base + u * (kReorderThreads / 8) + slot;
        if (p < a.n_tokens) *reinterpret_cast<uint4*>(dst + (int64_t)p * kHeadDim) = v[u];
        if (NORMS && t < 2) {   // the eight threads of a row are neighbouring lanes
            float x[8];
            unpack8(v[u], x);
            float s = 0.f;
#pragma unroll
            for (int e = 0; e < 8; ++e) s = fmaf(x[e], x[e], s);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            s += __shfl_xor_sync(0xffffffffu, s, 4);
            if (chunk == 0 && p < a.n_tokens) a.inv_norm[t][(int64_t)h * a.n_tokens + p] = fminf(rsqrtf(s), 1e12f);
        }
    }
}

cudaError_t launch_reorder(const ReorderArgs& a, cudaStream_t stream) {
    dim3 grid((a.n_tokens + kReorderTokensPerCta - 1) / kReorderTokensPerCta, a.heads, 3);
    if (a.inv_norm[0])
        return launch_kernel(reorder_kernel<true>, grid, kReorderThreads, 0, stream, a);
    return launch_kernel(reorder_kernel<false>, grid, kReorderThreads, 0, stream, a);
}

// ------------------------------------------------------------------------------------
// a2 under first-frame anchoring (the paper's appendix on error mitigation: all tokens of frame 0 are dst tokens), for the
//     blocks of the first frame group whose dst tokens exceed what match_team_kernel holds (a quarter of the largest block:
//     blocks of two or three frames).  Same rule, plain formulation: one CTA per (tensor, head, block), the block's rows
//     gathered through the reorder index into shared memory, inverse norms, for every src token the dot products with
//     the dst tokens (the block's first n_dst tokens) by fp32 FMAs on exact bf16 products, best dst (ties: lowest),
//     then the r best src by rank counting (ties: lowest position).  These blocks are 1 / (frame groups) of the scene.
// ------------------------------------------------------------------------------------
constexpr int kAnchorThreads = 128;
constexpr int kAnchorPitch = kRowBytes + 16;   // row pitch in shared memory: 16-byte accesses of neighbouring rows on distinct banks
__host__ __device__ constexpr int anchor_smem_bytes(int nmax) { return nmax * (kAnchorPitch + 12); }   // rows, inverse norms, scores, best dst

__global__ void __launch_bounds__(kAnchorThreads) match_anchor_kernel(const MatchArgs a, const TensorView src_q, const TensorView src_k,
                                                                       const int32_t* __restrict__ pi, int n_anchor, int main_capacity, int nmax) {
    extern __shared__ __align__(16) unsigned char sm_anchor[];
    depend_wait();
    dependents_launch();
    const int task = blockIdx.x;
    const int b = task % n_anchor, h = (task / n_anchor) % a.heads, t = task / (n_anchor * a.heads);
    const BlockInfo bi = a.blocks[b];
    const int n = bi.n, nd = t == 0 ? bi.nd_q : bi.nd_k, r = t == 0 ? bi.r_q : bi.r_k;
    if (bi.n_rule == n || nd <= main_capacity || r == 0 || n > nmax) return;   // the match kernel has written this block's map
    unsigned char* rows = sm_anchor;
    float* inv = reinterpret_cast<float*>(sm_anchor + (size_t)nmax * kAnchorPitch);
    float* score = inv + nmax;
    int* best = reinterpret_cast<int*>(score + nmax);
    const TensorView& sv = t == 0 ? src_q : src_k;
    const __nv_bfloat16* base = sv.ptr + (int64_t)h * sv.stride_head;
    for (int q = threadIdx.x; q < n * 8; q += kAnchorThreads) {
        const int row = q >> 3, c = q & 7;
        const int64_t orig = pi ? __ldg(pi + bi.start + row) : bi.start + row;   // (no index: the tensors are the reordered copies)
        *reinterpret_cast<uint4*>(rows + row * kAnchorPitch + c * 16) = ld_global(reinterpret_cast<const uint4*>(base + orig * sv.stride_token + c * 8));
    }
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += kAnchorThreads) {
        float ss = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            float x[8];
            unpack8(*reinterpret_cast<const uint4*>(rows + j * kAnchorPitch + c * 16), x);
#pragma unroll
            for (int e = 0; e < 8; ++e) ss = fmaf(x[e], x[e], ss);
        }
        inv[j] = fminf(rsqrtf(ss), 1e12f);   // 1 / max(|x|, 1e-12)
    }
    __syncthreads();
    for (int j = nd + threadIdx.x; j < n; j += kAnchorThreads) {   // src tokens: everything behind the block's tokens of frame 0
        float xs[64];
#pragma unroll
        for (int c = 0; c < 8; ++c) unpack8(*reinterpret_cast<const uint4*>(rows + j * kAnchorPitch + c * 16), xs + 8 * c);
        float top = -INFINITY;
        int arg = 0;
        for (int d = 0; d < nd; ++d) {
            float dot = 0.f;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                float xd[8];
                unpack8(*reinterpret_cast<const uint4*>(rows + d * kAnchorPitch + c * 16), xd);   // (the same row for every thread: a broadcast)
#pragma unroll
                for (int e = 0; e < 8; ++e) dot = fmaf(xs[8 * c + e], xd[e], dot);
            }
            const float sim = dot * inv[d];
            if (sim > top) {
                top = sim;
                arg = d;
            }
        }
        score[j] = top * inv[j];
        best[j] = arg;
    }
    __syncthreads();
    int32_t* A = a.assign[t] + (int64_t)h * a.n_tokens + bi.start;
    for (int j = threadIdx.x; j < n; j += kAnchorThreads) {
        if (j < nd) {
            A[j] = bi.start + j;
            continue;
        }
        const uint32_t key = score_key(score[j]);
        int rank = 0;   // src tokens that come before this one: better score, or the same score at a lower position
        for (int i = nd; i < n; ++i) {
            const uint32_t ki = score_key(score[i]);
            rank += (ki > key || (ki == key && i < j)) ? 1 : 0;
        }
        A[j] = bi.start + (rank < r ? best[j] : j);
    }
}

cudaError_t launch_match_anchor(const MatchArgs& a, const TensorView& src_q, const TensorView& src_k, const int32_t* pi, int n_anchor,
                                int main_capacity, int max_block_tokens, cudaStream_t stream) {
    if (n_anchor <= 0) return cudaSuccess;
    const int nmax = max_block_tokens < kMaxBlockTokens ? max_block_tokens : kMaxBlockTokens;
    return launch_kernel(match_anchor_kernel, 2 * a.heads * n_anchor, kAnchorThreads, anchor_smem_bytes(nmax), stream, a, src_q, src_k, pi, n_anchor, main_capacity, nmax);
}

cudaError_t launch_match(const MatchArgs& a, int max_block_tokens, int sm_count, cudaStream_t stream) {
    return max_block_tokens <= 64 ? launch_match_small(a, max_block_tokens, sm_count, stream) : launch_match_mid(a, max_block_tokens, sm_count, stream);
}
cudaError_t launch_merge(const MergeArgs& a, int max_block_tokens, int sm_count, cudaStream_t stream) {
    return max_block_tokens <= 32 ? launch_merge_small(a, sm_count, stream) : launch_merge_mid(a, max_block_tokens, sm_count, stream);
}

// ------------------------------------------------------------------------------------
// Adaptive outlier filtering for the query tokens (Sec. 3.4, Algorithm 2), blocks of at most 32 tokens.
//   deviation_kernel   eps[h][p] = || q_p - mean of the group p was merged into ||_2 (0 for a group of one)
//   threshold_kernel   tau = the (K+1)-th largest eps over all heads (K = the global budget): radix select
//   filter_kernel      outliers (eps > tau) leave their groups; the map is rewritten, the kept tokens of
//                      every (head, block) are counted
//   offsets_kernel     per head: merged row of every block's first kept token (prefix sum over the blocks),
//                      merged length, and the head's first 128-row query tile (for the attention kernel)
// ------------------------------------------------------------------------------------
__device__ void finish_level(const OutlierArgs& a, int level, int* hist);   // (threshold selection, below)
// Latency of the warps' instruction streams and bytes in flight bound the deviation kernel: as many warps as fit.  With one stage per warp (refilled while the
// distances are computed: a lane keeps its token in registers), 16 channels of the means at a time and a histogram of the 1024 bins that occur three CTAs fit on an SM; two
// stages and two CTAs, before: the five kernels of the filter 59.4 us at 32 976 tokens, now 55.3; the call 697.9 -> 693.8.  A grid of two CTAs per SM is never better, also where the third saves
// no round: calls at ratio 0.9 with two / three 61.5 / 59.2 us at 5 496 tokens, 96.6 / 94.4 at 10 992, 218.9 / 213.2 at 27 480, 371.6 / 362.5 at 43 968; 49.9 / 50.0 at 2 748.
constexpr int kDevWarps = 8;     // 8 x 8.5 KB of shared memory: three CTAs per SM
constexpr int kCentStride = 68;  // floats per mean: 16-byte reads of eight different means fall on distinct banks
constexpr int kDevAux = 16 * kCentStride * 4 + 16 * 4 + 32 + 64;   // means of the groups of two or more (at most 16 in 32 tokens), reciprocal sizes, an mbarrier, rows
constexpr int kDevBins = 1024;   // of level 0: the sign bit of a deviation is 0
constexpr int kDevSmem = kDevWarps * (32 * kRowBytes + kDevAux) + kDevBins * 4 /*histogram*/ + 1024 /*alignment slack*/;

__global__ void __launch_bounds__(kDevWarps * 32, 3)
deviation_kernel(const __grid_constant__ CUtensorMap map_q, const OutlierArgs a) {
    constexpr uint32_t STAGE_BYTES = 32 * kRowBytes;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + align_pad(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tq = lane & 3;   // MMA accumulator layout: rows g, g + 8; columns 2 tq, 2 tq + 1
    unsigned char* stage = smem + warp * STAGE_BYTES;
    unsigned char* aux = smem + kDevWarps * STAGE_BYTES + warp * kDevAux;
    float* cent = reinterpret_cast<float*>(aux);                   // [16][68] group means
    float* rcnt = cent + 16 * kCentStride;                         // [16] 1 / group size
    int* hist = reinterpret_cast<int*>(smem + kDevWarps * (STAGE_BYTES + kDevAux));   // [1024] bits 30-21 of this CTA's deviations
    for (int i = threadIdx.x; i < kDevBins; i += kDevWarps * 32) hist[i] = 0;
    __syncthreads();
    const uint32_t mbar = smem_u32(aux + 16 * kCentStride * 4 + 16 * 4), blk = smem_u32(stage);
    __nv_bfloat16* rows_of = reinterpret_cast<__nv_bfloat16*>(aux + 16 * kCentStride * 4 + 16 * 4 + 32);   // [32] mean of each token, in fragment order
    if (lane == 0) {
        mbar_init(mbar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    const SourceLayout& L = a.layout;
    const int box_f = min(L.blk_frames, L.frames), box_h = min(L.blk_h, L.grid_h), box_w = min(L.blk_w, L.grid_w);
    const int box_rows = box_f * box_h * box_w;
    const int own_t = lane / (box_h * box_w), own_y = (lane / box_w) % box_h, own_x = lane % box_w;
    for (int q = box_rows * 8 + lane; q < 32 * 8; q += 32)   // rows no load ever writes enter the MMAs with weight 0: keep them finite
        *reinterpret_cast<uint4*>(stage + q * 16) = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    BoxMap bm;
    bm.clipped = false;

    const int64_t n_tasks = (int64_t)a.heads * a.n_blocks;   // (head, block), queries only
    const int64_t stride = (int64_t)gridDim.x * kDevWarps;
    const int64_t first = (int64_t)blockIdx.x * kDevWarps + warp;
    TaskCursor cur, nxt;
    cur.init(first, stride, a.heads, a.n_blocks);   // one "tensor": t stays 0 while the task index is in range
    nxt = cur;
    auto issue = [&]() {   // lane 0 only
        const BlockGeom bg = a.geom[nxt.u];
        mbar_expect_tx(mbar, (uint32_t)box_rows * kRowBytes);
        tma_block_load(blk, &map_q, mbar, bg.x0, bg.y0, bg.s0, nxt.h);
    };
    if (!a.early) depend_wait();
    if (first < n_tasks && lane == 0) issue();
    nxt.advance();
    if (a.early) depend_wait();
    dependents_launch();

    uint32_t phase = 0;   // of the stage's barrier
    bool failed = false;
    for (int64_t task = first; task < n_tasks; task += stride, cur.advance(), nxt.advance(), phase ^= 1u) {
        const bool more = task + stride < n_tasks;
        const int h = cur.h;
        const BlockInfo bi = a.blocks[cur.u];
        const BlockGeom bg = a.geom[cur.u];
        bm.set(box_f, box_h, box_w, bg.frames, bg.rows, bg.cols);
        const int n = bi.n, r = bi.r_q;
        const int tok = (own_t < bg.frames && own_y < bg.rows && own_x < bg.cols) ? (own_t * bg.rows + own_y) * bg.cols + own_x : -1;
        float* eps = a.eps + (int64_t)h * a.n_tokens + bi.start;
        int rep = -1;   // stage ROW of the token this lane's token was merged into
        if (r > 0 && tok >= 0) {
            rep = ld_global(a.assign_q + (int64_t)h * a.n_tokens + bi.start + tok) - bi.start;
            if (rep < 0 || rep >= n) {
                atomicCAS(a.status, kDevOk, kDevBadIndex);
                rep = tok;
            }
            rep = bm.row_of_token(rep);
        }
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(mbar, phase, a.status, kDevTimeoutMatchLoad))) {
            failed = true;
            break;
        }
        if (r == 0) {   // nothing merged in this block: every deviation is 0
            if (tok >= 0) eps[tok] = 0.f;
            __syncwarp();
            if (more && lane == 0) issue();
        } else {
            // groups of two or more tokens get a mean; row of the mean = rank of the group's representative among them
            const unsigned group = __match_any_sync(0xffffffffu, rep);   // (lanes without a token share rep = -1: ignored below)
            const int group_size = rep >= 0 ? __popc(group) : 0;
            const unsigned multi = __ballot_sync(0xffffffffu, rep == lane && group_size >= 2);
            const int row_of = group_size >= 2 ? __popc(multi & ((1u << rep) - 1u)) : -1;
            if (rep == lane && group_size >= 2) rcnt[row_of] = 1.0f / (float)group_size;
            rows_of[fragment_order(lane)] = __float2bfloat16_rn((float)row_of);
            __syncwarp();   // rows and reciprocal group sizes visible
            // group sums = W x on the tensor cores, as in merge_small_kernel: W [16 means][32 tokens] of zeros and ones, 16 channels at a time; the means stay in
            // fp32 (no rounding to bf16 before the distance)
            const int n_ks = box_rows > 16 ? 2 : 1, n_cent = __popc(multi);
            uint32_t af[2][4];
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) w_fragment(af[ks], *reinterpret_cast<const uint2*>(rows_of + 16 * ks + 4 * tq), row_pair(g), row_pair(g + 8));
            const float i0 = g < n_cent ? rcnt[g] : 0.f, i1 = g + 8 < n_cent ? rcnt[g + 8] : 0.f;
            const uint32_t from = blk + (lane & 15) * kRowBytes;
#pragma unroll
            for (int np = 0; np < 4; ++np) {
                const uint32_t chunk = ((2 * np + (lane >> 4)) ^ (lane & 7)) << 4;
                uint32_t bf[2][4];
                float c[2][4];
                ldmatrix_x4_trans(bf[0], from + chunk);
                if (n_ks > 1) ldmatrix_x4_trans(bf[1], from + 16 * kRowBytes + chunk);
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    mma_first(c[nt], af[0], bf[0][2 * nt], bf[0][2 * nt + 1]);
                    if (n_ks > 1) mma_bf16_16816(c[nt], af[1], bf[1][2 * nt], bf[1][2 * nt + 1]);
                    float* to = cent + (2 * np + nt) * 8 + 2 * tq;
                    if (g < n_cent) *reinterpret_cast<float2*>(to + g * kCentStride) = make_float2(c[nt][0] * i0, c[nt][1] * i0);
                    if (g + 8 < n_cent) *reinterpret_cast<float2*>(to + (g + 8) * kCentStride) = make_float2(c[nt][2] * i1, c[nt][3] * i1);
                }
            }
            uint4 x8[8];   // this lane's token (stage row `lane`)
#pragma unroll
            for (int ch = 0; ch < 8; ++ch) x8[ch] = *reinterpret_cast<const uint4*>(stage + lane * kRowBytes + ((ch ^ (lane & 7)) << 4));
            __syncwarp();   // means visible, every lane has read the stage
            if (more && lane == 0) issue();
            float dev = 0.f;
            if (tok >= 0) {
                float2 d2 = make_float2(0.f, 0.f);   // even and odd channels
                if (row_of >= 0) {   // distance of this lane's token to its group's mean
                    const float* cr = cent + row_of * kCentStride;
#pragma unroll
                    for (int ch = 0; ch < 8; ++ch) {
                        float x[8];
                        unpack8(x8[ch], x);
                        const float4 lo = *reinterpret_cast<const float4*>(cr + ch * 8), hi = *reinterpret_cast<const float4*>(cr + ch * 8 + 4);
                        const float2 m[4] = {make_float2(lo.x, lo.y), make_float2(lo.z, lo.w), make_float2(hi.x, hi.y), make_float2(hi.z, hi.w)};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 d = tc::fsub2(make_float2(x[2 * e], x[2 * e + 1]), m[e]);
                            d2 = tc::ffma2(d, d, d2);
                        }
                    }
                }
                dev = sqrtf(d2.x + d2.y);
                eps[tok] = dev;
            }
            // level 0 of the threshold selection: histogram of the top 11 bits (zeros are not counted), one atomic per distinct bin
            const int bin = (int)(__float_as_uint(dev) >> 21) & (kDevBins - 1);
            const unsigned peers = __match_any_sync(0xffffffffu, bin);
            if (bin > 0 && lane == __ffs(peers) - 1) atomicAdd(&hist[bin], __popc(peers));
        }
        __syncwarp();   // every lane is done with the tables
    }
    if (failed) mbar_wait_bounded(mbar, phase, a.status, kDevTimeoutMatchLoad);   // give the copy in flight a bounded chance to land before the shared memory is released
    __syncthreads();
    for (int i = threadIdx.x; i < kDevBins; i += kDevWarps * 32) {
        const int c = hist[i];
        if (c) atomicAdd(a.sel + kSelHist + i, c);
    }
    finish_level(a, 0, reinterpret_cast<int*>(smem));   // (the stages, which nothing is copied to any more)
}

// ---- tau = the (K+1)-th largest deviation over all heads (K = the budget): radix select on the bit patterns of the
// non-negative floats (they order like the values), 11 + 11 + 10 bits.  Level 0's histogram is built by the
// deviation kernel while it writes the deviations; two refinement kernels rescan them (2 MB, resident in L2) for the
// elements inside the prefix chosen so far.  In each kernel the CTA that finishes last walks the histogram down from
// the largest bin until the remaining rank falls inside one, and leaves prefix and rank for the next level.
// Zeros are never counted at level 0: the walk ends in bin 0 whatever it holds.
// The chain of kernels is bound by latency, most of it the one CTA at each kernel's end.  With that CTA's loads in flight together, the walk
// over the bins and the table of query tiles spread over a warp's lanes, four loads in flight per thread in the refinement and one atomic per
// CTA on the count of outliers, the five kernels took 30 us instead of 39 (1 044 tokens x 16 heads), 39 instead of 47 (10 992), 60 instead of 68 (32 976).

// One warp: bin and remaining rank for histogram h[nb] (shared memory), as the sequential walk
//   above = 0; for (bin = nb - 1; bin > 0 && above + h[bin] <= rank; --bin) above += h[bin];  rank -= above
// It is the serial end of every level: a lane's run of bins (64, then the 2 of the run found; 32 and 1 with 1024 bins) is read in an order that
// has the lanes on different banks.
__device__ __forceinline__ void select_bin(const int* h, int nb, int rank, int* bin_out, int* rank_out) {
    const int lane = threadIdx.x & 31, per = nb >> 5, lo = lane * per;
    int c = 0;
#pragma unroll 8
    for (int i = 0; i < per; ++i) c += h[lo + ((i + lane) & (per - 1))];
    if (lane == 0) c -= h[0];   // bin 0 ends the walk: it is never added
    auto this_and_higher = [&](int v) {   // sum over this lane and all higher ones
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_down_sync(0xffffffffu, v, off);
            if (lane + off < 32) v += o;
        }
        return v;
    };
    const int incl = this_and_higher(c);
    const unsigned hit = __ballot_sync(0xffffffffu, incl > rank);
    if (hit == 0) {             // fewer than rank + 1 elements above bin 0
        if (lane == 0) {
            *bin_out = 0;
            *rank_out = rank - incl;
        }
        return;
    }
    const int run = 31 - __clz(hit);   // the walk stops inside this run of bins, above bin 0
    const int above_run = __shfl_sync(0xffffffffu, incl - c, run), two = nb >> 10;   // bins per lane
    const int b = run * per + lane * two;
    const int high = two == 2 ? h[b + 1] : 0, low = b > 0 ? h[b] : 0;
    const int incl2 = above_run + this_and_higher(high + low);
    if (lane == 31 - __clz(__ballot_sync(0xffffffffu, incl2 > rank))) {
        const int above = incl2 - low - high;
        const bool at_high = two == 2 && above + high > rank;
        *bin_out = at_high ? b + 1 : b;
        *rank_out = rank - (at_high ? above : above + high);
    }
}

// The bin of one level from its complete histogram (one CTA of 256 threads; hist: 2048 ints of shared memory).
__device__ void select_level(const OutlierArgs& a, int level, int* hist) {
    __shared__ int s_bin, s_rank;
    const int64_t count = a.total_count;
    if (level == 0 && (a.budget <= 0 || a.budget >= count)) {   // nothing is an outlier (tau = +inf) / everything is (tau = -1)
        if (threadIdx.x == 0) {
            *a.tau = a.budget <= 0 ? INFINITY : -1.0f;
            a.sel[kSelFinished] = 1;
        }
        return;
    }
    if (level > 0 && ld_global_cg(a.sel + kSelFinished)) return;
    const int nb = level == 2 ? 1024 : 2048, shift = level == 0 ? 21 : (level == 1 ? 10 : 0);
    int counts[8];   // (256 threads; all loads in flight before the first store)
#pragma unroll
    for (int u = 0; u < 8; ++u) counts[u] = u * 256 < nb ? ld_global_cg(a.sel + kSelHist + level * 2048 + u * 256 + threadIdx.x) : 0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
        if (u * 256 < nb) hist[u * 256 + threadIdx.x] = counts[u];
    __syncthreads();
    if (threadIdx.x < 32) {
        const int rank = level == 0 ? (int)a.budget : ld_global_cg(a.sel + kSelRank + level - 1);
        select_bin(hist, nb, rank, &s_bin, &s_rank);
        __syncwarp();
        if (threadIdx.x == 0) {
            const uint32_t prefix = (level == 0 ? 0u : (uint32_t)ld_global_cg(a.sel + kSelPrefix + level - 1)) | ((uint32_t)s_bin << shift);
            if (level < 2) {
                a.sel[kSelPrefix + level] = (int)prefix;
                a.sel[kSelRank + level] = s_rank;
            } else {
                *a.tau = __uint_as_float(prefix);
            }
        }
    }
}

// End of a level, called by every thread of every CTA after the CTA's histogram has been added to the global one:
// the CTA that arrives last selects the bin - unless the selection is deferred (head-sharded layers: the histograms
// of the other shards are still to be added; select_level_kernel runs behind the exchange).
__device__ void finish_level(const OutlierArgs& a, int level, int* hist) {
    __shared__ int s_last;
    if (a.defer_select) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(a.sel + kSelDone + level, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    select_level(a, level, hist);
}
__global__ void __launch_bounds__(256) select_level_kernel(const OutlierArgs a, int level) {
    __shared__ int hist[2048];
    depend_wait();
    dependents_launch();
    select_level(a, level, hist);
}

constexpr int kRefineThreads = 256;
static_assert(kRefineThreads == 256 && kDevWarps * 32 == 256, "select_level reads the histogram with 256 threads");
// LEVEL 1: histogram of bits 20-10 of the deviations whose bits 31-21 equal the level-0 choice; LEVEL 2: of bits 9-0
// of those whose bits 31-10 equal the choice so far.  LEVEL 0 (only where the deviation kernel does not build it on the
// fly: the large-block path): histogram of bits 31-21 of all deviations.
template <int LEVEL>
__global__ void __launch_bounds__(kRefineThreads) refine_kernel(const OutlierArgs a) {
    __shared__ int hist[2048];
    depend_wait();
    dependents_launch();
    if (ld_global(a.sel + kSelFinished)) return;   // (same answer in every thread of every CTA)
    constexpr int NB = LEVEL == 2 ? 1024 : 2048, SHIFT = LEVEL == 0 ? 21 : (LEVEL == 1 ? 10 : 0);
    constexpr uint32_t MASK = LEVEL == 0 ? 0u : (LEVEL == 1 ? 0xffe00000u : 0xfffffc00u);
    for (int i = threadIdx.x; i < NB; i += kRefineThreads) hist[i] = 0;
    __syncthreads();
    const uint32_t prefix = LEVEL == 0 ? 0u : (uint32_t)ld_global_cg(a.sel + kSelPrefix + (LEVEL > 0 ? LEVEL - 1 : 0));
    const int64_t count = (int64_t)a.heads * a.n_tokens, quads = count >> 2;
    const uint4* bits4 = reinterpret_cast<const uint4*>(a.eps);   // (the array comes from cudaMalloc: 16-byte aligned)
    auto tally = [&](uint32_t b) {
        if ((b & MASK) == prefix) atomicAdd(&hist[(b >> SHIFT) & (NB - 1)], 1);
    };
    const int64_t step = (int64_t)gridDim.x * kRefineThreads;
    for (int64_t i = (int64_t)blockIdx.x * kRefineThreads + threadIdx.x; i < quads; i += 4 * step) {   // four loads in flight
        uint4 b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) b[u] = i + u * step < quads ? ld_global(bits4 + i + u * step) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i + u * step < quads) {
                tally(b[u].x);
                tally(b[u].y);
                tally(b[u].z);
                tally(b[u].w);
            }
    }
    if (blockIdx.x == 0 && threadIdx.x < (int)(count & 3)) tally(__float_as_uint(a.eps[(quads << 2) + threadIdx.x]));
    __syncthreads();
    for (int i = threadIdx.x; i < NB; i += kRefineThreads) {
        const int c = hist[i];
        if (c) atomicAdd(a.sel + kSelHist + LEVEL * 2048 + i, c);
    }
    finish_level(a, LEVEL, hist);
}

// Outliers leave their groups (Sec. 3.4 item 4): one warp per (head, block), lane = token of the block.
// An outlier maps to itself; the other tokens of a group stay together, under their old representative if
// that is not an outlier, else under the remaining member with the lowest position.
__global__ void __launch_bounds__(256) filter_kernel(const OutlierArgs a) {
    depend_wait();
    dependents_launch();
    const int lane = threadIdx.x & 31;
    const int64_t task = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    __shared__ int s_out;   // outliers of this CTA: one atomic each on the count of all
    if (threadIdx.x == 0) s_out = 0;
    __syncthreads();
    if (task < (int64_t)a.heads * a.n_blocks) {
        const int h = (int)(task / a.n_blocks), b = (int)(task - (int64_t)h * a.n_blocks);
        const BlockInfo bi = a.blocks[b];
        const int n = bi.n;
        const float tau = *a.tau;
        const int32_t* A = a.assign_q + (int64_t)h * a.n_tokens + bi.start;
        int32_t* A_out = a.assign_q_out + (int64_t)h * a.n_tokens + bi.start;
        int rep = -1 - lane;   // lanes without a token match nobody
        bool outl = false;
        if (lane < n) {
            rep = A[lane] - bi.start;
            if (rep < 0 || rep >= n) {
                atomicCAS(a.status, kDevOk, kDevBadIndex);
                rep = lane;
            }
            outl = a.eps[(int64_t)h * a.n_tokens + bi.start + lane] > tau;
        }
        const unsigned out_mask = __ballot_sync(0xffffffffu, outl);
        const unsigned group = __match_any_sync(0xffffffffu, rep);
        int now = lane;
        if (lane < n && !outl) now = ((out_mask >> rep) & 1u) ? __ffs(group & ~out_mask) - 1 : rep;
        const unsigned kept = __ballot_sync(0xffffffffu, lane < n && now == lane);
        if (lane < n) A_out[lane] = bi.start + now;
        if (lane == 0) {
            a.kept_cnt[(int64_t)h * a.n_blocks + b] = __popc(kept);
            if (out_mask) atomicAdd(&s_out, __popc(out_mask));
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_out) atomicAdd(a.sel + kSelOutliers, s_out);
}

// Per head (one CTA each): merged row of every block's first kept token = specials + exclusive prefix sum of the kept
// counts, and the merged length.  The CTA that finishes last builds, over the heads, the index of each head's first
// 128-row query tile (for the attention kernel).
constexpr int kOffsetsThreads = 1024;
__global__ void __launch_bounds__(kOffsetsThreads, 1) offsets_kernel(const OutlierArgs a) {
    __shared__ int warp_sum[32];
    __shared__ int s_last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, h = blockIdx.x;
    depend_wait();
    dependents_launch();
    const int32_t* cnt = a.kept_cnt + (int64_t)h * a.n_blocks;
    int32_t* moff = a.moff_var + (int64_t)h * a.n_blocks;
    int running = a.n_special_total;
    int c_next = (int)threadIdx.x < a.n_blocks ? cnt[threadIdx.x] : 0;
    for (int b0 = 0; b0 < a.n_blocks; b0 += kOffsetsThreads) {
        const int b = b0 + threadIdx.x, c = c_next;
        c_next = b + kOffsetsThreads < a.n_blocks ? cnt[b + kOffsetsThreads] : 0;
        int incl = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += o;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        if (warp == 0) {   // inclusive scan of the 32 warp totals
            int w = warp_sum[lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, w, off);
                if (lane >= off) w += o;
            }
            warp_sum[lane] = w;
        }
        __syncthreads();
        if (b < a.n_blocks) moff[b] = running + (warp > 0 ? warp_sum[warp - 1] : 0) + incl - c;
        running += warp_sum[31];
        __syncthreads();   // the totals are read before the next chunk overwrites them
    }
    if (threadIdx.x == 0) {
        a.mq_head[h] = running;
        __threadfence();
        s_last = atomicAdd(a.sel + kSelOffsetsDone, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (s_last && warp == 0) {   // a lane per head (one thread that walked them took a load's latency for each)
        __threadfence();
        int t = 0;
        for (int h0 = 0; h0 < a.heads; h0 += 32) {
            const int tiles = h0 + lane < a.heads ? (ld_global_cg(a.mq_head + h0 + lane) + 127) / 128 : 0;
            int incl = tiles;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += o;
            }
            if (h0 + lane < a.heads) a.tile_prefix[h0 + lane] = t + incl - tiles;
            t += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) a.tile_prefix[a.heads] = t;
    }
}

cudaError_t launch_deviation(const OutlierArgs& a, int sm_count, cudaStream_t stream) {
    CUtensorMap mq;
    if (!encode_block_map(&mq, a.src_q, a.layout, a.heads)) return cudaErrorInvalidValue;
    const int64_t n_tasks = (int64_t)a.heads * a.n_blocks;
    int64_t grid = (n_tasks + kDevWarps - 1) / kDevWarps;
    if (grid > 3ll * sm_count) grid = 3ll * sm_count;
    if (grid < 1) grid = 1;
    return launch_kernel(deviation_kernel, (unsigned)grid, kDevWarps * 32, kDevSmem, stream, mq, a);
}
cudaError_t launch_threshold(const OutlierArgs& a, int sm_count, cudaStream_t stream) {
    const int64_t quads = ((int64_t)a.heads * a.n_tokens) >> 2;
    int64_t grid = (quads + kRefineThreads * 4 - 1) / (kRefineThreads * 4);   // about four 16-byte loads per thread
    if (grid > 2ll * sm_count) grid = 2ll * sm_count;
    if (grid < 1) grid = 1;
    cudaError_t e = launch_kernel(refine_kernel<1>, (unsigned)grid, kRefineThreads, 0, stream, a);
    if (e != cudaSuccess) return e;
    return launch_kernel(refine_kernel<2>, (unsigned)grid, kRefineThreads, 0, stream, a);
}
cudaError_t launch_threshold0(const OutlierArgs& a, int sm_count, cudaStream_t stream) {
    const int64_t quads = ((int64_t)a.heads * a.n_tokens) >> 2;
    int64_t grid = (quads + kRefineThreads * 4 - 1) / (kRefineThreads * 4);
    if (grid > 2ll * sm_count) grid = 2ll * sm_count;
    if (grid < 1) grid = 1;
    cudaError_t e = launch_kernel(refine_kernel<0>, (unsigned)grid, kRefineThreads, 0, stream, a);
    if (e != cudaSuccess) return e;
    return launch_threshold(a, sm_count, stream);
}
cudaError_t launch_refine_level(const OutlierArgs& a, int level, int sm_count, cudaStream_t stream) {
    const int64_t quads = ((int64_t)a.heads * a.n_tokens) >> 2;
    int64_t grid = (quads + kRefineThreads * 4 - 1) / (kRefineThreads * 4);
    if (grid > 2ll * sm_count) grid = 2ll * sm_count;
    if (grid < 1) grid = 1;
    if (level == 0)
        return launch_kernel(refine_kernel<0>, (unsigned)grid, kRefineThreads, 0, stream, a);
    if (level == 1)
        return launch_kernel(refine_kernel<1>, (unsigned)grid, kRefineThreads, 0, stream, a);
    return launch_kernel(refine_kernel<2>, (unsigned)grid, kRefineThreads, 0, stream, a);
}
cudaError_t launch_select_level(const OutlierArgs& a, int level, cudaStream_t stream) {
    return launch_kernel(select_level_kernel, 1, 256, 0, stream, a, level);
}
cudaError_t launch_offsets(const OutlierArgs& a, cudaStream_t stream) {
    return launch_kernel(offsets_kernel, (unsigned)a.heads, kOffsetsThreads, 0, stream, a);
}
cudaError_t launch_filter(const OutlierArgs& a, cudaStream_t stream) {
    const int64_t threads = (int64_t)a.heads * a.n_blocks * 32;
    cudaError_t e = launch_kernel(filter_kernel, (unsigned)((threads + 255) / 256), 256, 0, stream, a);
    if (e != cudaSuccess) return e;
    return launch_offsets(a, stream);
}

// ------------------------------------------------------------------------------------
// a5. Head-wise unmerge + inverse reorder + head concat (Eq. 5-7): every original token
//     copies the attention output of the merged query token it went into.
//     8 threads move one 128-byte (token, head) row.  A CTA works on one head and 128
//     consecutive original tokens: the map reads of neighbouring tokens share sectors and
//     the merged rows they point to are close together.  Each thread carries four rows at
//     a time so that four independent load chains are in flight.
// ------------------------------------------------------------------------------------
constexpr int kUnmergeThreads = 256;
constexpr int kUnmergeUnroll = 4;
constexpr int kUnmergeTokensPerCta = (kUnmergeThreads / 8) * kUnmergeUnroll;

__global__ void __launch_bounds__(kUnmergeThreads) unmerge_kernel(const __grid_constant__ UnmergeArgs a) {
    const int h = blockIdx.y;
    const int chunk = threadIdx.x & 7, slot = threadIdx.x >> 3;
    const int base = blockIdx.x * kUnmergeTokensPerCta;
    const int32_t* rank = a.rank_q + (int64_t)h * a.n_tokens;
    const uint4* om = reinterpret_cast<const uint4*>(a.o_m + (int64_t)h * a.m_q * kHeadDim) + chunk;
    __nv_bfloat16* out = a.out + (int64_t)h * a.out_stride_head + chunk * 8;
    int p[kUnmergeUnroll], row[kUnmergeUnroll];
    uint4 v[kUnmergeUnroll];
#pragma unroll
    for (int u = 0; u < kUnmergeUnroll; ++u) {
        const int i = base + u * (kUnmergeThreads / 8) + slot;
        p[u] = i < a.n_tokens ? __ldg(a.pi_inv + i) : 0;
    }
    if (!a.early) depend_wait();
#pragma unroll
    for (int u = 0; u < kUnmergeUnroll; ++u) row[u] = ld_global_cg(rank + p[u]);
    if (a.early) depend_wait();
    dependents_launch();
#pragma unroll
    for (int u = 0; u < kUnmergeUnroll; ++u) {
        if (row[u] < 0 || row[u] >= a.m_q) {   // corrupt map: record, copy row 0 instead of reading out of range
            atomicCAS(a.status, kDevOk, kDevBadIndex);
            row[u] = 0;
        }
        v[u] = ld_global(om + (int64_t)row[u] * 8);
    }
#pragma unroll
    for (int u = 0; u < kUnmergeUnroll; ++u) {
        const int i = base + u * (kUnmergeThreads / 8) + slot;
        if (i < a.n_tokens) *reinterpret_cast<uint4*>(out + (int64_t)i * a.out_stride_token) = v[u];
    }
}

cudaError_t launch_unmerge(const UnmergeArgs& a, cudaStream_t stream) {
    dim3 grid((a.n_tokens + kUnmergeTokensPerCta - 1) / kUnmergeTokensPerCta, a.heads);
    return launch_kernel(unmerge_kernel, grid, kUnmergeThreads, 0, stream, a);
}

cudaError_t configure_kernels() {
    cudaError_t e;
#define HTTM_SET_SMEM(kern, bytes)                                                                      \
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(bytes));          \
    if (e != cudaSuccess) return e;
    HTTM_SET_SMEM(deviation_kernel, kDevSmem);
#undef HTTM_SET_SMEM
    if ((e = configure_small_blocks()) != cudaSuccess || (e = configure_mid_blocks()) != cudaSuccess) return e;
    return configure_attention();
}

}  // namespace httm
