// Entry points shared between the library's translation units (not exported).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace trihost {

// Lets a kernel take up to `most` bytes of dynamic shared memory.  The limit belongs to
// the kernel and the device, not to a launch, and calls on other threads set it too:
// `most` is the same in every call, so that none lowers it between another's call
// and launch.
template <class K>
cudaError_t allow_smem(K *kernel, size_t most)
{
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e != cudaSuccess) (void)cudaGetLastError();  // reported by the caller's status alone
    return e;
}

// FP32 direct-difference EDM under any block map (edm.cu).
int edm_fp32(const float *x, uint32_t n, uint32_t d, float *out, int map, uint32_t rho, uint32_t reg,
             cudaStream_t s);

// Tensor-core Gram EDM with split FP16 operands and recompute of flagged pairs (edm_tc.cu).
size_t edm_tc_workspace(uint32_t n, uint32_t d, int prec);
int edm_tc(const float *x, uint32_t n, uint32_t d, float *out, int map, int prec, void *ws, size_t ws_bytes,
           unsigned long long *n_flagged, cudaStream_t s);

}  // namespace trihost
