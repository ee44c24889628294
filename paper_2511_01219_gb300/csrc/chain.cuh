// A batch's kernels run one after the other on one stream, each reading what the one before wrote.  They are launched as
// programmatic dependents: a kernel lets the next one start as soon as all of its own CTAs run (chain_go), and the next
// one waits at its first line until that kernel is complete and its writes are visible (chain_wait), so the launch itself
// and the placing of CTAs overlap the tail of the kernel before.  Between two ordinary launches the device idles 1.5 to
// 3 us, six times per batch.  A kernel launched with launch_chained calls both before it touches memory.
#pragma once
#include <cuda_runtime.h>

namespace relo {

__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace relo
