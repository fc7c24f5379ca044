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
    if (k) return k;
    if (slab_pow2(d, slab_threads(d))) return k_slab<FwdStage, PLAN_POW2, PLAN_POW2>;
    return k_slab<FwdStage, PLAN_ANY, PLAN_ANY>;
}
GroupKernel fwd_group_kernel(const SysDev &d, unsigned threads) {
    const int i2 = edge_index(d.K2), i3 = edge_index(d.K3);
    const GroupKernel k = i2 & 1 ? fwd_group_kernel_odd(i2, i3) : table().find_group(i2, i3);
    if (k) return k;
    if (slab_pow2(d, threads)) return k_slab_g<FwdStage, PLAN_POW2, PLAN_POW2>;
    return k_slab_g<FwdStage, PLAN_ANY, PLAN_ANY>;
}
cudaError_t configure_fwd_group_kernels() {
    for (cudaError_t e : {configure_fwd_group_kernels_odd(), table().configure_group(),
                          set_dynamic_smem((const void *)k_slab_g<FwdStage, PLAN_POW2, PLAN_POW2>, GROUP_SMEM_BYTES)})
        if (e != cudaSuccess) return e;
    return set_dynamic_smem((const void *)k_slab_g<FwdStage, PLAN_ANY, PLAN_ANY>, GROUP_SMEM_BYTES);
}

}  // namespace pme
