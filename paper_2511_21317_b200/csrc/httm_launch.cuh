// Kernel launches that overlap their prologue with the end of the kernel before them (programmatic dependent launch).
//
// A call is a chain of three to twelve kernels in one stream, each reading what the one before it wrote.  Launched the
// ordinary way, a kernel of a stream starts 1.5 - 2 us after its predecessor has ended, and then sets up its barriers, its
// tensor memory and its descriptors.  Every kernel of the library therefore lets its successor be launched as soon as all
// of its own CTAs run (dependents_launch), and does nothing but that set-up before depend_wait, which returns when
// the predecessor has completed and its writes are visible.  Because EVERY kernel waits, kernels that are further apart
// are ordered as well, and the one before the first may be anybody's (it then completes before ours start).
// Measured (calls back to back, before / after): 3 kernels on 1 044 tokens 26.7 / 23.1 us, 5 kernels on a ragged scene of
// 7 898 tokens 110 / 104 us, 9 kernels with outlier filtering on 32 976 tokens 750 / 736 us.
//
// What a kernel FURTHER back has written is complete even before depend_wait: the predecessor lets this kernel be launched only
// after its own wait.  Inside a call the merge and deviation kernels therefore start loading Q, K and V (which the match kernel
// waited for), and the unmerge kernel its map, while their predecessor still runs (`early` in their arguments; a kernel that is
// launched alone does not know what is in front of it and waits first).
// Measured (calls back to back, before / after): 1 044 tokens 21.0 / 20.5 us, 11 016 tokens 119.7 / 117.8, 7 898 tokens in clipped
// 48-token blocks 95.1 / 92.4, 32 976 tokens in 128-token blocks 167.2 / 159.5; with the filter's state cleared by the call's first
// kernel instead of a memset 32 976 tokens with outlier filtering 695.1 / 688.5.
//
// What the predecessor has written must be read by loads that stay behind the wait: ld_global below, or TMA.  __ldg reads
// through the non-coherent path, which assumes that the data does not change while the kernel runs, and is for the plan
// tables and other data that no kernel writes.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "httm_internal.h"

namespace httm {

__device__ __forceinline__ void depend_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependents_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ int32_t ld_global(const int32_t* p) {
    int32_t v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int32_t ld_global_cg(const int32_t* p) {   // from L2: written by other CTAs of the same kernel, or read ahead of depend_wait
    int32_t v;
    asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// zeros for the kernels behind this one (counters and histograms), spread over the CTAs: a memset of its own between two kernels would
// cost its launch and both overlaps
__device__ __forceinline__ void clear_words(const ClearRange (&clear)[2], int cta, int ctas) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (clear[k].words)
            for (int i = cta * (int)blockDim.x + (int)threadIdx.x; i < clear[k].n; i += ctas * (int)blockDim.x) clear[k].words[i] = 0;
}
__device__ __forceinline__ float ld_global(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ld_global(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

template <typename... Params, typename... Args>
cudaError_t launch_kernel(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace httm
