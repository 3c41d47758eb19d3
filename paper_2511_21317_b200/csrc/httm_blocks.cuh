// Device helpers of the kernels that work on one merging block per warp (httm_small_blocks.cu, httm_mem_kernels.cu): bounded
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

}  // namespace httm
