// Host interface of the grouped stage kernels (group.cu): every system of a group has the same mesh shape
// and B-spline order, so one launch per stage covers the whole group.
#pragma once

#include <cuda_runtime.h>

#include "kernels.h"

namespace pme {

struct GroupArgs {
    const SysDev *sys;  // the group's descriptors (device memory, nsys entries)
    int ips;            // work items per system of the launched stage
    int late;           // when the programmatic launch of the successor is triggered (PdlScope)
};

using GroupKernel = void (*)(GroupArgs);
// The grouped slab kernels for a system's plans and CTAs of that many threads, and the influence kernel (fwd.cu,
// conv.cu, inv.cu).
GroupKernel fwd_group_kernel(const SysDev &d, unsigned threads);
GroupKernel conv_group_kernel(const SysDev &d);
GroupKernel inv_group_kernel(const SysDev &d, unsigned threads);
// and the shared-memory limits of all of them.
cudaError_t configure_fwd_group_kernels();
cudaError_t configure_conv_group_kernels();
cudaError_t configure_inv_group_kernels();

#if defined(__CUDACC__)
// The CTA's system descriptor, copied from the group's array into shared memory.
__device__ __forceinline__ int group_load(const GroupArgs &a, SysDev &sd) {
    const int sys = blockIdx.x / a.ips;
    const int *src = (const int *)(a.sys + sys);
    for (int i = threadIdx.x; i < (int)(sizeof(SysDev) / 4); i += blockDim.x) ((int *)&sd)[i] = src[i];
    __syncthreads();
    return blockIdx.x - sys * a.ips;
}
#endif

// Raise the dynamic shared-memory limits of the grouped kernels (once per device).
cudaError_t configure_group_kernels();

// Work items of one system in a stage (binning: of this system's atoms).
int group_items(const SysDev &d, int stage);

// Enqueue the six stages for nsys systems whose descriptors are at sys_dev (device), all shaped like
// proto; max_nbin is the largest binning item count among them.
cudaError_t launch_group_chain(const SysDev *sys_dev, int nsys, const SysDev &proto, int max_nbin, cudaStream_t s);

}  // namespace pme
