// The inverse slab stage kernels (slab_kernels.cuh): those for every second K2 (inv2.cu has the others), the ones
// that pick their plans at run time, and the choice among them.
#include "slab_kernels.cuh"

namespace pme {

struct InvStage {
    template <int PR, int PC>
    static __device__ __forceinline__ void run(const SysDev &d, int k1, void *smem) {
        stage_inv<PR, PC>(d, k1, smem);
    }
};

static const SlabTable<InvStage, 0> &table() {
    static const SlabTable<InvStage, 0> t;
    return t;
}
StageKernel inv_kernel_odd(int i2, int i3);
GroupKernel inv_group_kernel_odd(int i2, int i3);
cudaError_t configure_inv_group_kernels_odd();

StageKernel inv_kernel(const SysDev &d) {
    const int i2 = edge_index(d.K2), i3 = edge_index(d.K3);
    const StageKernel k = i2 & 1 ? inv_kernel_odd(i2, i3) : table().find(i2, i3);
    return k ? k : k_slab<InvStage, -1, -1>;
}
GroupKernel inv_group_kernel(const SysDev &d) {
    const int i2 = edge_index(d.K2), i3 = edge_index(d.K3);
    const GroupKernel k = i2 & 1 ? inv_group_kernel_odd(i2, i3) : table().find_group(i2, i3);
    return k ? k : k_slab_g<InvStage, -1, -1>;
}
cudaError_t configure_inv_group_kernels() {
    for (cudaError_t e : {configure_inv_group_kernels_odd(), table().configure_group()})
        if (e != cudaSuccess) return e;
    return set_dynamic_smem((const void *)k_slab_g<InvStage, -1, -1>, GROUP_SMEM_BYTES);
}

}  // namespace pme
