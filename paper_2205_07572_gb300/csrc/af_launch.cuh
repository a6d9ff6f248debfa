// Launches whose CTAs may take their places on the SMs while the kernel before
// them in the stream is still finishing (programmatic dependent launch).
//
// The steps of a small grid and the substeps of an adaptive run are chains of
// short launches: without this, each began only when the one before had left
// the last SM, and its CTAs' start-up stood in the chain: acoustics on 512^2
// cells 14.3 us a step, 12.4 chained; 23 x 23 advection patches 36.9, 34.3 us.
//
// A kernel launched by launch_chained() calls chain_begin() before its first
// access to memory.  That waits until the kernel before it has completed and
// its writes are visible -- which holds for everything earlier in the stream
// too, as every chained kernel waits in every CTA before it can complete -- and
// then lets the next one's CTAs start.  Those are admitted when all CTAs of
// this kernel have begun, so they never take a place that one of them needs.
// It returns the CTA's index, read after the wait: addresses formed with it
// cannot be loaded from earlier, by whatever instruction (read-only loads are
// not held back by a memory clobber alone).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace af {

__device__ __forceinline__ unsigned chain_begin() {
    unsigned block;
    asm volatile("griddepcontrol.wait;\n griddepcontrol.launch_dependents;\n mov.u32 %0, %%ctaid.x;\n" : "=r"(block)::"memory");
    return block;
}

// chain = false: a launch like any other, after everything before it.  Kernels
// bound by the FP64 pipe take it: CTAs admitted early fill the SMs that happen
// to be free, and a launch of one wave is then as slow as its fullest SM
// (FP64 adaptive acoustics 679 us a coarse step, 688 chained).
template <typename... P, typename... Args>
inline cudaError_t launch_chained(bool chain, void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t stream, Args &&...args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = chain ? 1 : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // reported here, and not once more by whatever call reads the last error next
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, P(std::forward<Args>(args))...);
    const cudaError_t last = cudaGetLastError();
    return e != cudaSuccess ? e : last;
}

}  // namespace af
