// Device helpers of the kernels that work on merging blocks (httm_small_blocks.cu, httm_mid_blocks.cu, httm_mem_kernels.cu): bounded
// waits, block loads, warp-level matrix instructions, block geometry.
#pragma once

#include "httm_internal.h"
#include "tc_sm100.cuh"   // mbarrier / TMA wrappers (device), tensor-map encoders (host)

namespace httm {

// ------------------------------------------------------------------------------------
// small device helpers (mbarrier and address wrappers: tc_sm100.cuh)
// ------------------------------------------------------------------------------------
using tc::mbar_expect_tx;
using tc::mbar_init;
using tc::mbar_try_wait;
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return tc::smem_addr(p); }
// Bounded wait of the warp-per-block kernels: gives up after about two seconds, records `code` in the
// status word and returns false.  Never spins forever.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar, uint32_t parity, int32_t* status, int code) {
    if (mbar_try_wait(mbar, parity)) return true;
    const uint64_t t0 = tc::timer_ns();
    for (;;) {
        for (int i = 0; i < 64; ++i)
            if (mbar_try_wait(mbar, parity)) return true;
        if (tc::timer_ns() - t0 > 2000000000ull) {
            atomicCAS(status, kDevOk, code);
            return false;
        }
    }
}
__device__ __forceinline__ void unpack8(const uint4& raw, float* f) {
    f[0] = __uint_as_float(raw.x << 16);
    f[1] = __uint_as_float(raw.x & 0xffff0000u);
    f[2] = __uint_as_float(raw.y << 16);
    f[3] = __uint_as_float(raw.y & 0xffff0000u);
    f[4] = __uint_as_float(raw.z << 16);
    f[5] = __uint_as_float(raw.z & 0xffff0000u);
    f[6] = __uint_as_float(raw.w << 16);
    f[7] = __uint_as_float(raw.w & 0xffff0000u);
}

// ------------------------------------------------------------------------------------
// Task cursor: (tensor t, head h, unit u) of a linear task index that advances by a fixed
// stride, kept up to date with carries instead of 64-bit divisions in the loop.
// ------------------------------------------------------------------------------------
struct TaskCursor {
    int t, h, u;
    int st, sh, su;        // the stride, decomposed the same way
    int heads, units;
    __device__ void init(int64_t first, int64_t stride, int heads_, int units_) {
        heads = heads_;
        units = units_;
        const int64_t per_tensor = (int64_t)heads * units;
        t = (int)(first / per_tensor);
        int64_t rem = first - t * per_tensor;
        h = (int)(rem / units);
        u = (int)(rem - (int64_t)h * units);
        st = (int)(stride / per_tensor);
        rem = stride - st * per_tensor;
        sh = (int)(rem / units);
        su = (int)(rem - (int64_t)sh * units);
    }
    __device__ __forceinline__ void advance() {
        u += su;
        if (u >= units) {
            u -= units;
            ++h;
        }
        h += sh;
        if (h >= heads) {
            h -= heads;
            ++t;
        }
        t += st;
    }
};

// bytes to the next multiple of 1024.  Added to the shared array's own name, so that the compiler still knows the address space:
// behind a pointer rounded up as an integer every access was a generic one (a call on 11 016 tokens 121.0 -> 119.7 us, outlier
// filtering of 32 976 tokens 77.8 -> 72.1 us).
__device__ __forceinline__ uint32_t align_pad(const void* shared) { return (0u - smem_u32(shared)) & 1023u; }

// tiled TMA load {64 channels, rows, heads} -> this CTA's shared memory; the channel coordinate is 0
__device__ __forceinline__ void tma_rows_load(uint32_t dst_smem, const CUtensorMap* map, uint32_t mbar, int row, int head) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
                     dst_smem),
                 "l"(reinterpret_cast<uint64_t>(map)), "r"(mbar), "r"(0), "r"(row), "r"(head)
                 : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t* r, uint32_t saddr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(saddr)
                 : "memory");
}
// c (16x8 fp32) += a (16x16 bf16, row) * b (16x8 bf16, col)
__device__ __forceinline__ void mma_bf16_16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// tiled TMA load of one merging block straight from an original tensor: {64 channels, x, y, frame, head}
__device__ __forceinline__ void tma_block_load(uint32_t dst_smem, const CUtensorMap* map, uint32_t mbar, int x0, int y0, int s0, int head) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(dst_smem),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(mbar), "r"(0), "r"(x0), "r"(y0), "r"(s0), "r"(head)
        : "memory");
}
// Direct mode: a block arrives as the box [box_frames][box_h][box_w] of 128-byte rows (zero rows where the block
// is clipped by the grid edge or the last frame); its tokens are numbered in the same (frame, row, column)
// order without the holes.  For a block that is not clipped both numberings coincide.
struct BoxMap {
    int box_h, box_w;          // rows and columns of the box
    int rows, cols;            // of this block
    uint32_t m_plane, m_cols;  // multipliers for floor(j / (rows * cols)) and floor(j / cols), j < 256
    bool clipped;
    __device__ void set(int box_frames, int bh, int bw, int frames, int r, int c) {
        box_h = bh;
        box_w = bw;
        rows = r;
        cols = c;
        clipped = frames != box_frames || r != bh || c != bw;
        if (clipped) {
            m_plane = 65536u / (uint32_t)(r * c) + 1u;
            m_cols = 65536u / (uint32_t)c + 1u;
        }
    }
    // token number -> box row
    __device__ __forceinline__ int row_of_token(int j) const {
        if (!clipped) return j;
        const int t = (int)(((uint32_t)j * m_plane) >> 16), rem = j - t * rows * cols;
        const int y = (int)(((uint32_t)rem * m_cols) >> 16), x = rem - y * cols;
        return (t * box_h + y) * box_w + x;
    }
};
// monotone map float -> uint32 (larger float <-> larger key); every real score maps to a key >= 1
__device__ __forceinline__ uint32_t score_key(float s) {
    const uint32_t b = __float_as_uint(s);
    return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}

__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t* r, uint32_t saddr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(saddr)
                 : "memory");
}

// 5-D map of the patch tokens of an original tensor with one merging block as the box
inline bool encode_block_map(CUtensorMap* map, const TensorView& t, const SourceLayout& L, int heads) {
    const int bw = L.blk_w < L.grid_w ? L.blk_w : L.grid_w, bh = L.blk_h < L.grid_h ? L.blk_h : L.grid_h,
              bf = L.blk_frames < L.frames ? L.blk_frames : L.frames;
    return encode_patch_tensor_map(map, t.ptr + (int64_t)L.n_special * t.stride_token, L.grid_w, L.grid_h, L.frames, heads, t.stride_token,
                                   L.tokens_per_frame, t.stride_head, bw, bh, bf);
}

// (head, unit of the head) of a linear index that advances by a fixed stride
struct UnitCursor {
    int h, u, sh, su, units;
    __device__ void init(int first, int stride, int units_) {
        units = units_;
        h = first / units;
        u = first - h * units;
        sh = stride / units;
        su = stride - sh * units;
    }
    __device__ __forceinline__ void advance() {
        h += sh;
        u += su;
        if (u >= units) {
            u -= units;
            ++h;
        }
    }
};

// Host: CTAs of eight warps per SM, 2 or 3, for kernels whose warps work off a unit at a time.  The third pays where it saves more than a third of the rounds.  Calls on 32-token
// blocks, 16 heads, ratio 0.9, with two CTAs / three (rounds in brackets): 5 496 tokens (2 / 1) 34.6 / 32.1 us, 16 488 (5 / 3) 80.3 / 78.6; where it saves less, 10 992 (3 / 2) 56.1 / 57.0,
// 13 740 (4 / 3) 69.1 / 69.8, 19 236 (5 / 4) 112.3 / 117.5, 27 480 (7 / 5) 158.9 / 161.2.  From six rounds of 24 warps on the merge kernel takes 2 - 4 % less with three (32 976 tokens
// 56.3 / 54.1, 65 952 105.5 / 103.4), the calls are within 1 % either way: 30 228 (8 / 6) 175.2 / 177.0, 32 976 (9 / 6) 190.7 / 189.5, at ratio 0.7 578 / 566, 43 968 (12 / 8) 280.1 / 281.7,
// 65 952 (17 / 12) 516 / 518.
inline int unit_ctas(int64_t units, int sm_count) {
    const int64_t warps = 8ll * (sm_count < 1 ? 1 : sm_count), rounds2 = (units + 2 * warps - 1) / (2 * warps), rounds3 = (units + 3 * warps - 1) / (3 * warps);
    return rounds3 > 5 || 3 * rounds3 < 2 * rounds2 ? 3 : 2;
}

struct Geometry {   // BlockGeom in registers
    int s0, y0, x0, frames, rows, cols;
};
__device__ __forceinline__ int4 load_geometry(const BlockGeom* geom, int u) { return __ldg(reinterpret_cast<const int4*>(geom + u)); }
__device__ __forceinline__ Geometry unpack_geometry(const int4& v) {
    Geometry g;
    g.s0 = (int16_t)(v.x & 0xffff);
    g.y0 = v.x >> 16;
    g.x0 = (int16_t)(v.y & 0xffff);
    g.frames = v.y >> 16;
    g.rows = (int16_t)(v.z & 0xffff);
    g.cols = v.z >> 16;
    return g;
}
// frames, rows and columns of a block in bits of their own (each is at most 256).  What the match kernels keep from block to block holds for
// one shape, so the key has to tell all shapes apart: blocks clipped in time and in width, (1, 4, 4) and (4, 4, 1), have equally many tokens.
__device__ __forceinline__ int shape_key(const int4& v) { return (v.z & 0x3ff) | (v.z >> 16) << 10 | (v.y >> 16) << 20; }
// d (16x8 fp32) = a (16x16 bf16, row) * b (16x8 bf16, col): the first step of a sum
__device__ __forceinline__ void mma_first(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}
// floor(x / d) for 0 <= x < 2^20, d >= 1: (x + 0.5) / d is at least 0.5 / d away from an integer, more than the error x / d * 2^-22 of the
// approximate quotient
__device__ __forceinline__ int small_div(int x, int d) { return (int)__fdividef((float)x + 0.5f, (float)d); }
struct Box {   // extents of a block's TMA box (the block shape, clipped to the scene)
    int frames, h, w, rows;
    __device__ void set(const SourceLayout& L) {
        frames = min(L.blk_frames, L.frames);
        h = min(L.blk_h, L.grid_h);
        w = min(L.blk_w, L.grid_w);
        rows = frames * h * w;
    }
};
// stage row of token j of a block
__device__ __forceinline__ int row_of_token(const Box& box, const Geometry& g, int j) {
    if (g.rows == box.h && g.cols == box.w) return j;   // (frames come last: clipping them leaves the numbering alone)
    const int plane = g.rows * g.cols, t = small_div(j, plane), rem = j - t * plane, y = small_div(rem, g.cols);
    return (t * box.h + y) * box.w + rem - y * g.cols;
}
// token number of stage row rho, -1 if the row holds none
__device__ __forceinline__ int token_of_row(const Box& box, const Geometry& g, int rho) {
    if (g.rows == box.h && g.cols == box.w) return rho < g.frames * box.h * box.w ? rho : -1;
    const int line = small_div(rho, box.w), t = small_div(line, box.h), y = line - t * box.h, x = rho - line * box.w;
    return t < g.frames && y < g.rows && x < g.cols ? (t * g.rows + y) * g.cols + x : -1;
}

__device__ __forceinline__ float inv_norm(float square) {   // 1 / max(|x|, 1e-12), within 2 ulp
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(square));
    return fminf(r, 1e12f);
}

// Two numbers of merged rows as bf16 each (whole numbers up to 256 are exact) against two others: 1.0 where equal, else 0.  That IS a
// register of the fragment of W, the 0/1 matrix of merged rows x tokens; put together from integer comparisons it took four times
// the instructions (merging 32-token blocks of 32 976 tokens 64.5 -> 62.4 us).  Tables of them have the 16 tokens of a step in fragment order: 2 q, 2 q + 1, 2 q + 8, 2 q + 9 for q = 0 .. 3.
__device__ __forceinline__ uint32_t equal_rows(uint32_t rows, uint32_t row) {
    const __nv_bfloat162 e = __heq2(*reinterpret_cast<const __nv_bfloat162*>(&rows), *reinterpret_cast<const __nv_bfloat162*>(&row));
    return *reinterpret_cast<const uint32_t*>(&e);
}
__device__ __forceinline__ int fragment_order(int token) { return (token & ~15) + 4 * ((token & 7) >> 1) + 2 * ((token >> 3) & 1) + (token & 1); }
__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// fragment of W (16 merged rows x 16 tokens): rw = merged rows of this lane's four tokens, b0 and b1 its own two rows (row_pair)
__device__ __forceinline__ uint32_t row_pair(int row) { return pack2_bf16((float)row, (float)row); }
__device__ __forceinline__ void w_fragment(uint32_t* af, const uint2& rw, uint32_t b0, uint32_t b1) {
    af[0] = equal_rows(rw.x, b0);
    af[1] = equal_rows(rw.x, b1);
    af[2] = equal_rows(rw.y, b0);
    af[3] = equal_rows(rw.y, b1);
}

// DIRECT: the blocks come straight from the original tensors (5-D block maps), the special tokens frame by
// frame (4-D frame maps); otherwise from the reordered copies, specials in chunks of 32.
struct MergeMaps {
    CUtensorMap block[3], special[3];
};

// Host: the tensor maps of a merge launch.  Blocks from the original tensors or runs of box_rows rows of the reordered copies.
inline bool encode_merge_maps(MergeMaps* m, const MergeArgs& a, int box_rows) {
    const int64_t N = a.n_tokens;
    for (int t = 0; t < 3; ++t) {
        if (a.geom) {
            if (!encode_block_map(&m->block[t], a.src[t], a.layout, a.heads)) return false;
            m->special[t] = m->block[t];   // (not used without special tokens)
            if (a.layout.n_special > 0 &&
                !encode_frame_tensor_map(&m->special[t], a.src[t].ptr, a.layout.tokens_per_frame, a.layout.frames, a.heads, a.src[t].stride_token,
                                         a.src[t].stride_head, a.layout.n_special))
                return false;
        } else {
            if (!encode_rows_tensor_map(&m->block[t], a.xr[t], N, a.heads, kHeadDim, N * kHeadDim, box_rows)) return false;
            m->special[t] = m->block[t];   // not used
        }
    }
    return true;
}

}  // namespace httm
