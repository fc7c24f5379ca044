// The influence stage kernels, for one system and for a group of systems (batches, server waves): one per mesh
// edge K1 with its lane plan at compile time, and one that picks the plan at run time for the edges without.
#include <cuda_runtime.h>

#include "group.h"
#include "kernels.h"
#include "pdl.cuh"
#include "stages.cuh"

namespace pme {

// Four CTAs per SM: at K1 = 128 156 registers would leave three, and three waves of its 1040 items instead of two
// (20.5 -> 18.4 us; 128^3 evaluation 122.8 -> 120.7 us).
template <int P1>
__global__ void __launch_bounds__(NT_CONV, 4) k_conv(SysDev d) {
    extern __shared__ __align__(16) unsigned char smem[];
    PdlScope pdl(d.pdl_late);
    stage_conv<P1>(d, d.item0 + blockIdx.x, smem);
}

template <int P1>
__global__ void __launch_bounds__(NT_CONV, 4) k_conv_g(GroupArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SysDev sd;
    PdlScope pdl(a.late);
    const int item = group_load(a, sd);
    stage_conv<P1>(sd, item, smem);
}

StageKernel conv_kernel(const SysDev &d) {
#define PME_PICK(K) \
    if (d.lp_k1 == Edge<K>::P1) return k_conv<Edge<K>::P1>;
    PME_EDGES(PME_PICK)
#undef PME_PICK
    return k_conv<-1>;
}
GroupKernel conv_group_kernel(const SysDev &d) {
#define PME_PICK(K) \
    if (d.lp_k1 == Edge<K>::P1) return k_conv_g<Edge<K>::P1>;
    PME_EDGES(PME_PICK)
#undef PME_PICK
    return k_conv_g<-1>;
}

cudaError_t configure_conv_group_kernels() {
    cudaError_t e;
#define PME_CFG_K(K) \
    if ((e = set_dynamic_smem((const void *)k_conv_g<Edge<K>::P1>, GROUP_SMEM_BYTES)) != cudaSuccess) return e;
    PME_EDGES(PME_CFG_K)
#undef PME_CFG_K
    return set_dynamic_smem((const void *)k_conv_g<-1>, GROUP_SMEM_BYTES);
}

}  // namespace pme
