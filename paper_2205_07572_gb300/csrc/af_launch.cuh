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

#include <atomic>
#include <utility>

#include "af_internal.h"

namespace af {

__device__ __forceinline__ unsigned chain_begin() {
    unsigned block;
    asm volatile("griddepcontrol.wait;\n griddepcontrol.launch_dependents;\n mov.u32 %0, %%ctaid.x;\n" : "=r"(block)::"memory");
    return block;
}

// CTAs of Kern that an SM holds (0: the query failed).  One shared-memory size
// per kernel.
template <auto Kern>
inline int resident_ctas(int threads, size_t smem) {
    static std::atomic<int> held{0};
    int r = held.load(std::memory_order_relaxed);
    if (r == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, Kern, threads, smem) != cudaSuccess) {
            cudaGetLastError();  // not the launch's error
            r = 0;
        }
        held.store(r, std::memory_order_relaxed);
    }
    return r;
}

// True if a chain of grids of `grid` CTAs, `resident` to an SM, keeps its SMs
// evenly loaded: the next grid's CTAs take the places that the current one
// leaves, which are those of the SMs with the least of the current one.  That
// is harmless if all of them fit beside it, or if no SM can hold more than an
// even share; between the two some SMs end up with more, and a grid takes as
// long as its fullest SM: FP64 advection of 240 tiles of 32 x 32 cells 47 us,
// 67 chained; FP32 acoustics of 600 tiles of 16 x 16 9.0 and 11.5; swirl in FP64
// up to 1.5x.  (Twelve hundred chains measured: outside this range none was
// more than 7 % slower than unchained, most were 2 to 12 % faster.)
inline bool chain_even(int64_t grid, int resident) {
    return 2 * grid <= (int64_t)kSMs * resident || grid > (int64_t)kSMs * (resident - 1);
}

// The same where the grids in a row differ, so that the places left say nothing
// about the next grid's share: one CTA an SM, or more than the SMs can hold of
// them in uneven numbers.
inline bool chain_even_mixed(int64_t grid, int resident) {
    return grid <= kSMs || grid > (int64_t)kSMs * (resident - 1);
}

// True while `stream` records a graph.  What a chain hides is the gap between
// two launches, 3 us and more in a stream and 1 us in a graph: short kernels
// gain from it in a stream even where chain_even is false.
inline bool recording(cudaStream_t stream) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &st) != cudaSuccess) cudaGetLastError();
    return st == cudaStreamCaptureStatusActive;
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
