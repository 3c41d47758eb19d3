// The projections around the path (Algorithm 1's first and last lines: Q, K, V = x W_qkv and out = Attn W_o) as a
// tcgen05 GEMM of the library's own:  y[n][out] = x[n][in] . w[out][in]^T,  bf16 operands, fp32 accumulation in tensor
// memory, bf16 result.  Weights are given as [out][in] (the layout a linear layer stores them in), so both operands are
// K-major.
//
// Two CTAs (a cluster, on the two SMs of a TPC) work on one 256 x 256 output tile with tcgen05.mma.cta_group::2: each holds
// 128 rows of x and 128 rows of w of a 64-channel stage, and the tensor cores of both read both halves of w.  A CTA on
// its own with 128 x 256 tiles reads 48 KB of shared memory and 48 KB of L2 per 128 x 256 x 64 of work, a pair 32 KB per CTA;
// the operand traffic is what bounded a single CTA's kernel.  Measured, 1024 -> 3072: 10 992 rows 61.2 -> 48.9 us (1413
// TFLOP/s = 86 % of cuBLAS's burst rate on 8192^3), 65 952 rows 367 -> 285 us (1457).  It is bound by the power limit when
// run for longer (59 us) and by 7 rounds of tiles for 6.97 of work at the smaller size.
//   warp 0      TMA producer (in both CTAs): a ring of (x half tile, w half tile) stages, 128-byte swizzle; both halves
//               count on the leader's barrier
//   warp 1      in the leader (cluster rank 0): issues every MMA into one of two 256-column accumulators, in both CTAs
//   warps 2-5   epilogue (in both CTAs, 128 rows each): accumulator -> bf16 -> shared memory -> TMA store of 32 x 64 pieces
//               (whole lines; the tensor map clips at the last row and column), while the MMAs of the next tile run
// Persistent; consecutive clusters take the output tiles of the same 256 rows of x, so that x is read from DRAM once and the
// weights stay in L2.  Every wait is bounded; on expiry the status word is set and the kernel returns.
#include "../../include/httm.h"
#include "httm_internal.h"
#include "httm_launch.cuh"
#include "tc_sm100.cuh"

namespace httm {

namespace {

constexpr int BM = 128, BN = 256, BK = 64;   // rows of x per CTA (256 per pair), columns of the tile, channels per stage
constexpr int LIN_STAGES = 6;
constexpr int A_BYTES = BM * BK * 2, B_BYTES = (BN / 2) * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;   // 16 + 16 KB per CTA
constexpr int LIN_THREADS = 192;
constexpr int OUT_ROWS = 32, OUT_COLS = 64, OUT_BYTES = OUT_ROWS * OUT_COLS * 2;   // one store: 4 KB
constexpr int LIN_OFF_OUT = LIN_STAGES * STAGE_BYTES;                              // 4 warps x 2 buffers
constexpr int LIN_OFF_BARS = LIN_OFF_OUT + 8 * OUT_BYTES;
constexpr int LIN_SMEM = LIN_OFF_BARS + 256 + 1024 /*alignment slack*/;
static_assert(LIN_SMEM <= 227 * 1024, "shared memory of a CTA");

struct LinBars {
    uint64_t full[LIN_STAGES], empty[LIN_STAGES];   // full: the leader's are used
    uint64_t acc_full[2], acc_empty[2];             // acc_empty: the leader's are used
    uint32_t tmem_base;
    int abort_flag;
};

// address of the same shared-memory location in the cluster's CTA `rank`
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// bounded wait with cluster scope (arrivals come from the peer CTA too)
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const uint64_t t0 = tc::timer_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i) {
            uint32_t ok;
            asm volatile(
                "{\n\t.reg .pred p;\n\t"
                "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}"
                : "=r"(ok)
                : "r"(bar), "r"(parity)
                : "memory");
            if (ok) return true;
        }
        if (*abort_flag) return false;
        if (tc::timer_ns() - t0 > 2000000000ull) {
            *abort_flag = 1;
            return false;
        }
    }
}
// tile load into this CTA's shared memory that counts on a barrier of the pair (cluster address; c0 is 0)
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, uint32_t cluster_bar, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(cluster_bar), "r"(0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src),
                 "r"(c0), "r"(c1)
                 : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// one arrival on the barrier at this offset in BOTH CTAs when every MMA issued so far is done
__device__ __forceinline__ void commit_pair(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
                 "h"((uint16_t)3)
                 : "memory");
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(LIN_THREADS, 1)
linear_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_y,
              int n_rows, int out_features, int k_blocks, int n_tiles, int64_t total_tiles, int32_t* status) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t s0 = tc::smem_addr(smem);   // (the same offset in both CTAs: the kernel has no other shared memory)
    LinBars* bars = reinterpret_cast<LinBars*>(smem + LIN_OFF_BARS);
    volatile int* abort_flag = &bars->abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = blockIdx.x & 1u;     // cluster rank: clusters are pairs of consecutive CTAs

    if (tid == 0) {
        bars->abort_flag = 0;
        for (int i = 0; i < LIN_STAGES; ++i) {
            tc::mbar_init(tc::smem_addr(&bars->full[i]), 1);
            tc::mbar_init(tc::smem_addr(&bars->empty[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(tc::smem_addr(&bars->acc_full[i]), 1);
            tc::mbar_init(tc::smem_addr(&bars->acc_empty[i]), 8);   // one arrival per epilogue warp of the pair
        }
        tc::fence_barrier_init();
        tc::prefetch_tensormap(&map_x);
        tc::prefetch_tensormap(&map_w);
        tc::prefetch_tensormap(&map_y);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_addr(&bars->tmem_base)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc::fence_before_sync();
    __syncthreads();
    cluster_sync();   // the peer's barriers are initialised
    tc::fence_after_sync();
    const uint32_t tmem = bars->tmem_base;
    depend_wait();
    dependents_launch();

    const int64_t first = blockIdx.x >> 1, step = gridDim.x >> 1;   // this pair's output tiles
    if (warp == 0) {
        // ------------------------------------------------------------------ producer
        if (tc::elect_one()) {
            uint32_t cnt = 0;   // stages filled so far
            bool ok = true;
            for (int64_t t = first; ok && t < total_tiles; t += step) {
                const int m0 = (int)(t / n_tiles) * (2 * BM) + (int)rank * BM, n0 = (int)(t % n_tiles) * BN + (int)rank * (BN / 2);
                for (int kb = 0; kb < k_blocks; ++kb, ++cnt) {
                    const uint32_t st = cnt % LIN_STAGES, ph = (cnt / LIN_STAGES) & 1u;
                    ok = tc::mbar_wait(tc::smem_addr(&bars->empty[st]), ph ^ 1u, abort_flag);
                    if (!ok) break;
                    const uint32_t own = tc::smem_addr(&bars->full[st]), bar = map_to_rank(own, 0);
                    if (rank == 0) tc::mbar_expect_tx(own, 2 * STAGE_BYTES);   // of both CTAs; rows past the end are zero filled and counted
                    tma_load_3d_pair(s0 + st * STAGE_BYTES, &map_x, bar, m0, kb);
                    tma_load_3d_pair(s0 + st * STAGE_BYTES + A_BYTES, &map_w, bar, n0, kb);
                }
            }
            // the leader's arrivals on this CTA's barriers must have landed before the CTA leaves
            for (uint32_t i = 0; ok && i < LIN_STAGES; ++i, ++cnt)
                ok = tc::mbar_wait(tc::smem_addr(&bars->empty[cnt % LIN_STAGES]), ((cnt / LIN_STAGES) & 1u) ^ 1u, abort_flag);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (rank == 0 && tc::elect_one()) {
            constexpr uint32_t idesc = tc::idesc_bf16(2 * BM, BN, false, false);
            const uint64_t d0 = tc::smem_desc_sw128(s0);
            uint32_t cnt = 0, tile_i = 0;
            bool ok = true;
            for (int64_t t = first; ok && t < total_tiles; t += step, ++tile_i) {
                const uint32_t acc = tile_i & 1u;
                ok = mbar_wait_cluster(tc::smem_addr(&bars->acc_empty[acc]), ((tile_i >> 1) & 1u) ^ 1u, abort_flag);
                if (!ok) break;
                tc::fence_after_sync();
                for (int kb = 0; kb < k_blocks; ++kb, ++cnt) {
                    const uint32_t st = cnt % LIN_STAGES, ph = (cnt / LIN_STAGES) & 1u;
                    ok = mbar_wait_cluster(tc::smem_addr(&bars->full[st]), ph, abort_flag);
                    if (!ok) break;
                    tc::fence_after_sync();
                    const uint64_t da = d0 + (uint64_t)st * (STAGE_BYTES >> 4), db = da + (A_BYTES >> 4);
#pragma unroll
                    for (int k = 0; k < 4; ++k)   // four K = 16 steps of the 64-channel stage (32 bytes = 2 descriptor units each)
                        mma_pair(tmem + acc * BN, da + 2 * k, db + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
                    commit_pair(tc::smem_addr(&bars->empty[st]));   // the stage may be refilled when these MMAs are done
                }
                if (ok) commit_pair(tc::smem_addr(&bars->acc_full[acc]));
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ epilogue: lane = row of the warp's 32 rows
        const int quad = warp & 3;   // tensor memory lanes 32 quad .. belong to this warp
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        unsigned char* stage = smem + LIN_OFF_OUT + quad * 2 * OUT_BYTES;
        uint32_t tile_i = 0;
        for (int64_t t = first; t < total_tiles; t += step, ++tile_i) {
            const uint32_t acc = tile_i & 1u;
            const int row0 = (int)(t / n_tiles) * (2 * BM) + (int)rank * BM + quad * 32, n0 = (int)(t % n_tiles) * BN;
            if (!__all_sync(0xffffffffu, mbar_wait_cluster(tc::smem_addr(&bars->acc_full[acc]), (tile_i >> 1) & 1u, abort_flag))) break;
            tc::fence_after_sync();
#pragma unroll 1
            for (int c = 0; c < BN / OUT_COLS; ++c) {
                uint32_t r[OUT_COLS];
                tc::tmem_ld32(tmem + acc * BN + c * OUT_COLS + lane_addr, r);
                tc::tmem_ld32(tmem + acc * BN + c * OUT_COLS + 32 + lane_addr, r + 32);
                tc::tmem_wait_ld();
                if (c == BN / OUT_COLS - 1) {   // everything is in registers: the accumulator may be overwritten
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(map_to_rank(tc::smem_addr(&bars->acc_empty[acc]), 0));
                }
                unsigned char* buf = stage + (c & 1) * OUT_BYTES;
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");   // the store before the last has read this buffer
                __syncwarp();
#pragma unroll
                for (int q = 0; q < 8; ++q) {   // 16-byte piece q of the row sits at q ^ (row & 7)
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const __nv_bfloat162 p = __floats2bfloat162_rn(__uint_as_float(r[8 * q + 2 * e]), __uint_as_float(r[8 * q + 2 * e + 1]));
                        w[e] = *reinterpret_cast<const uint32_t*>(&p);
                    }
                    *reinterpret_cast<uint4*>(buf + lane * (OUT_COLS * 2) + ((q ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    if (row0 < n_rows && n0 + c * OUT_COLS < out_features) tma_store_2d(&map_y, tc::smem_addr(buf), n0 + c * OUT_COLS, row0);
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
    }
    tc::fence_before_sync();
    __syncthreads();
    cluster_sync();   // no arrival from the peer is still to come, its MMAs no longer touch this CTA's tensor memory
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    if (tid == 0 && bars->abort_flag) atomicCAS(status, kDevOk, kDevTimeoutLinear);
}

}  // namespace

cudaError_t configure_linear() { return cudaFuncSetAttribute(linear_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, LIN_SMEM); }

// Returns cudaErrorInvalidValue if a tensor map cannot be encoded.
cudaError_t launch_linear(const LinearArgs& a, int sm_count, cudaStream_t stream) {
    CUtensorMap mx, mw, my;
    // a matrix [rows][in] as {64 channels, rows, in / 64 blocks of 64 channels}: the block index is the third coordinate
    const int k_blocks = a.in_features / BK;
    const int64_t ldy = a.n_rows == 1 ? a.out_features : a.ldy;   // (not used then: it need not be a stride that a tensor map can hold)
    if (!encode_rows_tensor_map(&mx, a.x, a.n_rows, k_blocks, a.ldx, BK, BM) ||
        !encode_rows_tensor_map(&mw, a.w, a.out_features, k_blocks, a.ldw, BK, BN / 2) ||
        !encode_matrix_tensor_map(&my, a.y, a.n_rows, a.out_features, ldy, OUT_ROWS, OUT_COLS))
        return cudaErrorInvalidValue;
    const int n_tiles = (a.out_features + BN - 1) / BN;
    const int64_t total = ((a.n_rows + 2 * BM - 1) / (2 * BM)) * n_tiles;
    int pairs = sm_count < 2 ? 1 : sm_count / 2;
    if (pairs > total) pairs = (int)total;
    if (pairs < 1) return cudaSuccess;   // nothing to do
    return launch_kernel(linear_kernel, 2 * pairs, LIN_THREADS, LIN_SMEM, stream, mx, mw, my, (int)a.n_rows, a.out_features, k_blocks, n_tiles, total, a.status);
}

}  // namespace httm
