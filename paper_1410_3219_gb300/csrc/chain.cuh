// Kernels of one stream that follow each other closely.  In a small simulation
// a step is a chain of some twenty kernels of 4 to 20 us, and the gap between
// one's end and the next one's first instruction is a good part of it.  A
// kernel launched as a programmatic dependent is set up while the one before
// it still runs, and waits for that one's end (and for its writes) where it
// calls chained().  Every kernel of the chain calls it before it touches
// memory, so the order is that of the plain launches.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace rich {

constexpr int kSMs = 152;  // of a GB300

// From this many cells on kernels are launched plainly: the next one's
// waiting blocks would take the room of the running one's.  A step (with the
// mesh update) takes in dependent and in plain launches, FP64: 96 and 108 us for
// 8,100 cells, 178 and 194 for 65,536, 303 and 295 for 131,044, 515 and 485 for
// 262,144; split: 85 and 106, 135 and 150, 187 and 204, 286 and 277 (176,400:
// 211 and 230).  The line lies between the two precisions' own.
constexpr int64_t kChainedBelow = 1 << 17;

#ifdef __CUDACC__
// (cells: the number that launch_chained was given.  The two instructions do
// nothing in a plain launch, but are not free in a kernel of many blocks of one
// warp: the split-precision geometry at 1,048,576 cells took 252 us with them,
// 217 us without)
__device__ __forceinline__ void chained(int64_t cells)
{
    if (cells >= kChainedBelow) return;
    // let the next kernel be set up, then wait for the one before
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
#endif

template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), int grid, int block, cudaStream_t st, int64_t cells, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cells < kChainedBelow ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace rich
