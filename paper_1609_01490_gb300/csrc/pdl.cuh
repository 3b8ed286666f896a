// Launches of a call's own kernels back to back (programmatic dependent launch).
// The second kernel's blocks may start as soon as every block of the first has
// started (and called dependents_may_start) instead of after its last store has
// drained; they wait in wait_for_previous before they touch anything that the
// first writes or reads.  It saves 2 to 3 us a pair of launches: a collision call on
// 9001 discs takes 18.6 us (21.5 in stream order), a cost-model step 18.8 (20.4).
// A waiting block keeps its place: the blocks of the second kernel gather on the
// SMs that the first leaves early, so work that only a few blocks have is spread.
// Only between kernels of one call on one stream: the first is launched in the
// ordinary way, so that it follows everything before it in the stream, and each of the
// others waits before it touches anything that an earlier one writes or reads, so
// that a chain of them keeps its order.  A kernel launched so never reads an earlier
// one's results through const __restrict__ pointers or __ldg: such loads may be moved
// ahead of the wait, or come from a cache filled before it.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <utility>

namespace tri {

// Lets the next kernel's blocks start once every block has called this or ended.
__device__ __forceinline__ void dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Waits until the previous kernel has ended and its stores are visible; returns
// at once in a kernel launched in the ordinary way.
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace tri

namespace trihost {

template <class... P, class... A>
cudaError_t launch_behind(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
    if (e != cudaSuccess) (void)cudaGetLastError();  // the caller's to report, not the next launch's
    return e;
}

}  // namespace trihost
