// Kernel launches whose start overlaps the end of the kernel before them.
//
// A solver iteration is a chain of some 20 kernels, of which those on the coarse levels (and all of a
// small problem's) run for 2 to 6 us. Launched into a chained queue (programmatic dependent launch), a
// kernel's blocks are placed as soon as its predecessor's have ended, before its memory is flushed and
// its end reported; they read what no kernel of the chain writes (row pointers, columns), then wait for
// that in chain_wait(). 1-3% of a pass. Letting the next kernel be placed earlier still, while blocks of
// this one run (griddepcontrol.launch_dependents), made passes 2-7% slower instead: its waiting blocks
// take the slots and caches of the running ones.
#pragma once
#include <cuda_runtime.h>

#include "common.h"

namespace knp {

// A stream, and whether kernels launched into it may start before their predecessor has ended. Only the
// solver's own graphs are captured through a chained queue: every kernel in them calls chain_wait(), so
// the end of a kernel implies the end of all before it, and the programmatic edges stay out of a
// caller's capture.
struct Queue {
    cudaStream_t st;
    bool chained;
    Queue(cudaStream_t s, bool c = false) : st(s), chained(c) {}
};

// In the kernel: waits until the kernel before this one has ended and its writes are visible. What an
// earlier kernel of the chain writes is read only after it, through pointers without __restrict__, whose
// loads the compiler neither moves up nor sends through the read-only path. Without a chained launch it
// does nothing.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
void launch(void (*kernel)(P...), int64_t grid, int block, const Queue& q, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.stream = q.st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = q.chained ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    if (e != cudaSuccess) KNP_FAIL(KNP_ERR_CUDA, "kernel launch failed: %s", cudaGetErrorString(e));
}

}  // namespace knp
