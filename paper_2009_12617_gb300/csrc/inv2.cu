// The inverse slab stage kernels for every second K2 (slab_kernels.cuh), beside inv.cu.
#include "slab_kernels.cuh"

namespace pme {

struct InvStage {
    template <int PR, int PC>
    static __device__ __forceinline__ void run(const SysDev &d, int k1, void *smem) {
        stage_inv<PR, PC>(d, k1, smem);
    }
};

static const SlabTable<InvStage, 1> &table() {
    static const SlabTable<InvStage, 1> t;
    return t;
}
StageKernel inv_kernel_odd(int i2, int i3) { return table().find(i2, i3); }
GroupKernel inv_group_kernel_odd(int i2, int i3) { return table().find_group(i2, i3); }
cudaError_t configure_inv_group_kernels_odd() { return table().configure_group(); }

}  // namespace pme
