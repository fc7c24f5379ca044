// Stage kernels over a group of systems that share one mesh shape (K1, K2, K3, p): one launch per stage
// covers every work item of every system in the group, CTA b taking item b mod ips of system b / ips. The
// stage bodies and block sizes are the single-system ones, so a system's results are bit-identical to its
// single-system evaluation. Batches run one chain of six such launches per group, the chains as parallel
// branches of one CUDA graph.
#include <cuda_runtime.h>

#include "group.h"
#include "pdl.cuh"
#include "stages.cuh"

namespace pme {

__global__ void __launch_bounds__(NT_BIN) k_bin_g(GroupArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SysDev sd;
    PdlScope pdl(a.late);
    const int item = group_load(a, sd);
    if (item < sd.nbin) stage_bin(sd, item, smem);
}

template <int P, int T>
__global__ void __launch_bounds__(tile_nt_bound(T)) k_spread_g(GroupArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SysDev sd;
    spread_clear<P, T>(smem);  // before the wait: shared memory only
    PdlScope pdl(a.late);
    const int item = group_load(a, sd);
    stage_spread<P, T>(sd, item, smem, true);
}

template <int P, int T>
__global__ void __launch_bounds__(tile_nt_bound(T)) k_gather_g(GroupArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SysDev sd;
    PdlScope pdl(a.late);
    const int item = group_load(a, sd);
    stage_gather<P, T>(sd, item, smem);
}

// The spread / force kernels of a group: order p, tile edge 2^tlog.
template <int T>
static void (*spread_g_t(int p))(GroupArgs) {
    return p == 4 ? k_spread_g<4, T> : (p == 5 ? k_spread_g<5, T> : (p == 6 ? k_spread_g<6, T> : k_spread_g<8, T>));
}
template <int T>
static void (*gather_g_t(int p))(GroupArgs) {
    return p == 4 ? k_gather_g<4, T> : (p == 5 ? k_gather_g<5, T> : (p == 6 ? k_gather_g<6, T> : k_gather_g<8, T>));
}
static void (*spread_g(const SysDev &d))(GroupArgs) { return d.tlog == 4 ? spread_g_t<16>(d.p) : spread_g_t<8>(d.p); }
static void (*gather_g(const SysDev &d))(GroupArgs) { return d.tlog == 4 ? gather_g_t<16>(d.p) : gather_g_t<8>(d.p); }

cudaError_t configure_group_kernels() {
    for (int p : {4, 5, 6, 8})
        for (const void *f : {(const void *)spread_g_t<8>(p), (const void *)spread_g_t<16>(p),
                              (const void *)gather_g_t<8>(p), (const void *)gather_g_t<16>(p)}) {
            cudaError_t e = set_dynamic_smem(f, GROUP_SMEM_BYTES);
            if (e != cudaSuccess) return e;
        }
    for (cudaError_t e : {configure_fwd_group_kernels(), configure_conv_group_kernels(), configure_inv_group_kernels()})
        if (e != cudaSuccess) return e;
    return set_dynamic_smem((const void *)k_bin_g, GROUP_SMEM_BYTES);
}

int group_items(const SysDev &d, int stage) {
    switch (stage) {
        case STAGE_BIN: return d.nbin > 0 ? d.nbin : 1;
        case STAGE_SPREAD: return d.ntiles + OVF_ITEMS;
        case STAGE_FWD: return d.K1;
        case STAGE_CONV: return d.nconv;
        case STAGE_INV: return d.K1;
        default: return d.ntiles + OVF_ITEMS;
    }
}

template <class... Args>
static cudaError_t launch_ex(void (*kernel)(Args...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                             Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = launch_mode() ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

cudaError_t launch_group_chain(const SysDev *sys_dev, int nsys, const SysDev &proto, int max_nbin, cudaStream_t s) {
    GroupArgs a;
    a.sys = sys_dev;
    const SysDev &d = proto;
    const unsigned slab_nt = slab_group_threads(d, nsys);
    cudaError_t e;
    for (int stage = 0; stage < NUM_STAGES; ++stage) {
        a.late = pdl_when(launch_mode(), stage, d);
        a.ips = stage == STAGE_BIN ? (max_nbin > 0 ? max_nbin : 1) : group_items(d, stage);
        const unsigned grid = (unsigned)(a.ips * nsys);
        switch (stage) {
            case STAGE_BIN: e = launch_ex(k_bin_g, grid, NT_BIN, smem_bin(NT_BIN), s, a); break;
            case STAGE_SPREAD:
                e = launch_ex(spread_g(d), grid, (unsigned)tile_threads(d, (int64_t)max_nbin * BIN_CHUNK),
                              smem_spread(d.p, d.tlog), s, a);
                break;
            case STAGE_FWD: e = launch_ex(fwd_group_kernel(d, slab_nt), grid, slab_nt, smem_slab(d.K2, d.K3), s, a); break;
            case STAGE_CONV: e = launch_ex(conv_group_kernel(d), grid, NT_CONV, smem_conv(d.K1, NT_CONV), s, a); break;
            case STAGE_INV: e = launch_ex(inv_group_kernel(d, slab_nt), grid, slab_nt, smem_inv(d.K2, d.K3), s, a); break;
            default:
                e = launch_ex(gather_g(d), grid, (unsigned)tile_threads(d, (int64_t)max_nbin * BIN_CHUNK, true),
                              smem_gather_all(d.p, d.tlog), s, a);
                break;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace pme
