// The forward slab stage kernels for every second K2 (slab_kernels.cuh), beside fwd.cu.
#include "slab_kernels.cuh"

namespace pme {

struct FwdStage {
    template <int PR, int PC>
    static __device__ __forceinline__ void run(const SysDev &d, int k1, void *smem) {
        stage_fwd<PR, PC>(d, k1, smem);
    }
};

static const SlabTable<FwdStage, 1> &table() {
    static const SlabTable<FwdStage, 1> t;
    return t;
}
StageKernel fwd_kernel_odd(int i2, int i3) { return table().find(i2, i3); }
GroupKernel fwd_group_kernel_odd(int i2, int i3) { return table().find_group(i2, i3); }
cudaError_t configure_fwd_group_kernels_odd() { return table().configure_group(); }

}  // namespace pme
