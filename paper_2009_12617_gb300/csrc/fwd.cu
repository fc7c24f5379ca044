// The forward slab stage kernels (slab_kernels.cuh): those for every second K2 (fwd2.cu has the others), the ones
// that pick their plans at run time, and the choice among them.
#include "slab_kernels.cuh"

namespace pme {

struct FwdStage {
    template <int PR, int PC>
    static __device__ __forceinline__ void run(const SysDev &d, int k1, void *smem) {
        stage_fwd<PR, PC>(d, k1, smem);
    }
};

static const SlabTable<FwdStage, 0> &table() {
    static const SlabTable<FwdStage, 0> t;
    return t;
}
StageKernel fwd_kernel_odd(int i2, int i3);
GroupKernel fwd_group_kernel_odd(int i2, int i3);
cudaError_t configure_fwd_group_kernels_odd();

StageKernel fwd_kernel(const SysDev &d) {
    const int i2 = edge_index(d.K2), i3 = edge_index(d.K3);
    const StageKernel k = i2 & 1 ? fwd_kernel_odd(i2, i3) : table().find(i2, i3);
    return k ? k : k_slab<FwdStage, -1, -1>;
}
GroupKernel fwd_group_kernel(const SysDev &d) {
    const int i2 = edge_index(d.K2), i3 = edge_index(d.K3);
    const GroupKernel k = i2 & 1 ? fwd_group_kernel_odd(i2, i3) : table().find_group(i2, i3);
    return k ? k : k_slab_g<FwdStage, -1, -1>;
}
cudaError_t configure_fwd_group_kernels() {
    for (cudaError_t e : {configure_fwd_group_kernels_odd(), table().configure_group()})
        if (e != cudaSuccess) return e;
    return set_dynamic_smem((const void *)k_slab_g<FwdStage, -1, -1>, GROUP_SMEM_BYTES);
}

}  // namespace pme
