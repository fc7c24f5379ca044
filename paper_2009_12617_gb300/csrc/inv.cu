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
    if (k) return k;
    if (slab_pow2(d, slab_threads(d))) return k_slab<InvStage, PLAN_POW2, PLAN_POW2>;
    return k_slab<InvStage, PLAN_ANY, PLAN_ANY>;
}
GroupKernel inv_group_kernel(const SysDev &d, unsigned threads) {
    const int i2 = edge_index(d.K2), i3 = edge_index(d.K3);
    const GroupKernel k = i2 & 1 ? inv_group_kernel_odd(i2, i3) : table().find_group(i2, i3);
    if (k) return k;
    if (slab_pow2(d, threads)) return k_slab_g<InvStage, PLAN_POW2, PLAN_POW2>;
    return k_slab_g<InvStage, PLAN_ANY, PLAN_ANY>;
}
cudaError_t configure_inv_group_kernels() {
    for (cudaError_t e : {configure_inv_group_kernels_odd(), table().configure_group(),
                          set_dynamic_smem((const void *)k_slab_g<InvStage, PLAN_POW2, PLAN_POW2>, GROUP_SMEM_BYTES)})
        if (e != cudaSuccess) return e;
    return set_dynamic_smem((const void *)k_slab_g<InvStage, PLAN_ANY, PLAN_ANY>, GROUP_SMEM_BYTES);
}

}  // namespace pme
