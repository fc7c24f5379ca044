// The inverse slab stage kernels, for one system and for a group of systems (batches, server waves): one kernel per
// mesh edge K2 = K3 with that edge's lane plans at compile time (each holds only its plans' code, which keeps it
// small enough for the instruction caches), and one that picks the plans at run time for other meshes.
#include <cuda_runtime.h>

#include "group.h"
#include "kernels.h"
#include "pdl.cuh"
#include "stages.cuh"

namespace pme {

template <int PR, int PC>
__global__ void __launch_bounds__(NT_SLAB) k_inv(SysDev d) {
    extern __shared__ __align__(16) unsigned char smem[];
    PdlScope pdl(d.pdl_late);
    stage_inv<PR, PC>(d, d.item0 + blockIdx.x, smem);
}

template <int PR, int PC>
__global__ void __launch_bounds__(NT_SLAB) k_inv_g(GroupArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SysDev sd;
    PdlScope pdl(a.late);
    const int item = group_load(a, sd);
    stage_inv<PR, PC>(sd, item, smem);
}

#define PME_PICK(K, kernel) \
    if (d.lp_rows == Edge<K>::PR && d.lp_cols == Edge<K>::PC) return kernel<Edge<K>::PR, Edge<K>::PC>;
StageKernel inv_kernel(const SysDev &d) {
#define PME_PICK_K(K) PME_PICK(K, k_inv)
    PME_EDGES(PME_PICK_K)
#undef PME_PICK_K
    return k_inv<-1, -1>;
}
GroupKernel inv_group_kernel(const SysDev &d) {
#define PME_PICK_K(K) PME_PICK(K, k_inv_g)
    PME_EDGES(PME_PICK_K)
#undef PME_PICK_K
    return k_inv_g<-1, -1>;
}

cudaError_t configure_inv_group_kernels() {
    cudaError_t e;
#define PME_CFG_K(K) \
    if ((e = set_dynamic_smem((const void *)k_inv_g<Edge<K>::PR, Edge<K>::PC>, GROUP_SMEM_BYTES)) != cudaSuccess) return e;
    PME_EDGES(PME_CFG_K)
#undef PME_CFG_K
    return set_dynamic_smem((const void *)k_inv_g<-1, -1>, GROUP_SMEM_BYTES);
}

}  // namespace pme
