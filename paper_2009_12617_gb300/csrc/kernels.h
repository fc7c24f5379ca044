// Host-side interface of the CUDA kernels (launch configuration and entry points).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "common.cuh"

namespace pme {

constexpr int GB300_SMS = 152;

// The kernels have no other transforms than the lane plans': every accepted mesh has one for each direction.
constexpr bool every_mesh_has_plans() {
    for (int i = 0; i < N_EDGES; ++i) {
        if (conv_lane_plan(mesh_edge(i)) < 0) return false;
        for (int j = 0; j < N_EDGES; ++j)
            if (slab_lane_plan(mesh_edge(j) / 2, mesh_edge(i)) < 0 || slab_lane_plan(mesh_edge(i), mesh_edge(j) / 2 + 1) < 0) return false;
    }
    return true;
}
static_assert(every_mesh_has_plans(), "a mesh edge without lane plans");

constexpr int NT_BIN = 128;    // threads per CTA for binning (BIN_CHUNK atoms per CTA)
// Threads of the slab CTAs: SLAB_THREADS, or as many more (up to NT_SLAB) as let both passes run in one round of
// lanes (the plans are chosen to fit SLAB_THREADS where they can; long edges do not). 108^3, whose passes take 704 and
// 896 lanes: 70.0 -> 61.9 us an evaluation. A kernel's launch bound is its own count: all bounded at 1024, 64^3 ran
// 27.6 -> 28.9 us.
constexpr int NT_SLAB = 1024;
PME_HD int slab_nt(int pr, int pc) {  // lane plans of the rows (K3/2 points) and the columns (K2 points)
    const int K2 = plan_L(pc) * plan_E(pc), H3 = plan_L(pr) * plan_E(pr) + 1;
    const int rows = plan_units(pr, K2), cols = plan_units(pc, H3), most = rows > cols ? rows : cols;
    return most < SLAB_THREADS ? SLAB_THREADS : (most > NT_SLAB ? NT_SLAB : most);
}
inline unsigned slab_threads(const SysDev &d) { return (unsigned)slab_nt(d.lp_rows, d.lp_cols); }
// The same for a group of systems with `slabs` slabs in all. Where there are more than one per SM, several CTAs have to
// share an SM: SLAB_THREADS for slabs of up to SLAB_GROUP_POINTS points. us a batch of eight systems of 0.1 atoms a
// point with slab_nt / SLAB_THREADS: 80^3 220 / 211, 80 x 80 x 96 268 / 254, 64 x 64 x 128 233 / 221, 96^3 354 / 339,
// 100^3 418 / 401, but 108^3 525 / 547 and 128^3 804 / 810; of two systems: 80^3 82 / 80, 96^3 111 / 108, but 64 x 128 x 64
// (128 slabs) 78 / 87.
constexpr int SLAB_GROUP_POINTS = 10000;
PME_HD int slab_group_nt(int pr, int pc, int slabs) {
    const int K2 = plan_L(pc) * plan_E(pc), K3 = 2 * plan_L(pr) * plan_E(pr);
    return slabs > GB300_SMS && K2 * K3 <= SLAB_GROUP_POINTS ? SLAB_THREADS : slab_nt(pr, pc);
}
inline unsigned slab_group_threads(const SysDev &d, int nsys) { return (unsigned)slab_group_nt(d.lp_rows, d.lp_cols, nsys * d.K1); }
constexpr int NT_TILE = 256;   // threads per CTA for spreading and force interpolation (two per atom), at most,
constexpr int NT_TILE16 = 512; // with 8^3 / 16^3 tiles
PME_HD int tile_nt_bound(int T) { return T >= 16 ? NT_TILE16 : NT_TILE; }
// Spread / gather CTA size for a system whose binned atoms number about n_bins * BIN_CHUNK: two threads per
// atom, sized to the mean tile occupancy, so sparse 8^3 tiles (large meshes) do not leave half the CTA idle
// and twice as many CTAs fit on an SM. Dense 8^3 tiles interpolate forces on 192 threads: at 64 registers,
// five such CTAs fit on an SM, three beside an inverse-stage CTA that has not retired yet, so all tiles of
// a 64^3 mesh are dispatched at once (with 256 threads, 13-15 SMs ran a fifth tile in a second wave; 28.65
// vs 28.75 us per evaluation). 16^3 tiles (hundreds of atoms each) spread on 512 threads. Their force interpolation
// takes 512 threads too where there are few tiles per SM, so that each ends soon (p = 8, 80 x 80 x 96, 150 tiles: 73 us
// per evaluation against 88 with 256 or 128 threads); 256 at orders 5 and 6 with few atoms a tile, whose 512 threads
// would idle (90 x 96 x 100, 25000 atoms, p = 6: 53 against 58 with 512); and 128 where more than three tiles per SM (of
// 152) at orders 6 and 8 would come in waves (106 registers at p = 6: four 128-thread CTAs per SM but only one of 512;
// 128^3, 262144 atoms, p = 6: 126 against 129 with 256 and 131 with 512). Results do not depend on it.
inline int tile_threads(const SysDev &d, int64_t n, bool gather = false) {
    if (d.nt_tile == 128 || d.nt_tile == NT_TILE || (d.nt_tile == NT_TILE16 && d.tlog >= 4))
        return d.nt_tile;  // chosen by the autotuner or the caller
    if (d.tlog >= 4) {
        if (!gather) return NT_TILE16;
        if (d.p >= 6 && d.ntiles > 3 * GB300_SMS) return 128;
        return (d.p == 5 || d.p == 6) && n < (int64_t)200 * d.ntiles ? 256 : NT_TILE16;
    }
    if (d.ntiles > 0 && n <= (int64_t)64 * d.ntiles) return 128;
    return gather ? 192 : NT_TILE;
}
constexpr int NT_CONV = 128;   // threads per CTA for the influence stage
constexpr size_t MAX_SMEM_BYTES = 226 * 1024;  // opt-in limit is 227 KB including static shared memory
constexpr size_t GROUP_SMEM_BYTES = MAX_SMEM_BYTES - sizeof(SysDev) - 64;  // beside the system's descriptor

// Mesh edges K1 = K whose lane plan gets an influence kernel specialised at compile time.
#define PME_EDGES(X)                                                                                             \
    X(16) X(18) X(20) X(24) X(30) X(32) X(36) X(40) X(48) X(50) X(54) X(60) X(64) X(72) X(80) X(90) X(96) X(100) \
        X(108) X(120) X(128)
template <int K>
struct Edge {
    static constexpr int PR = slab_lane_plan(K / 2, K), PC = slab_lane_plan(K, K / 2 + 1), P1 = conv_lane_plan(K);
    static_assert(PR >= 0 && PC >= 0 && P1 >= 0, "every listed edge has lane plans");
};

// Launch mode of the per-stage kernels: 0 plain, 1 programmatic dependent launch triggered at kernel entry,
// 2 triggered at CTA exit (see pdl_when for the influence stage), 3 triggered right after the kernel's own wait.
// Process-wide; affects launches recorded afterwards.
void set_launch_mode(int mode);
int launch_mode();
// The PdlScope argument of a kernel of stage `stage` of system d in launch mode `mode`. In mode 2 a stage releases
// its successor at CTA exit, except the influence stage of meshes with K1 <= 64, which releases the inverse stage
// right after its own wait: those few slab CTAs fit beside the influence CTAs and are resident when they finish
// (evaluations of single graphs at 64^3 32.4 -> 32.0 us, 48^3 20.6 -> 20.4). More or larger slabs get in the way of the
// influence CTAs (with / without the early release: 80^3 45.2 / 41.3 us an evaluation, 96^3 52.1 / 45.7, 108^3
// 80.2 / 70.0, 96 x 90 x 108 81.7 / 75.2). Other stages' successors were slower or no faster when released early.
int pdl_when(int mode, int stage, const SysDev &d);

// CTAs per slab of the single-system forward and inverse slab stages: 1, or 2 / 4 (a thread-block cluster
// per slab exchanging its intermediate rows / columns through distributed shared memory; meshes with
// K2 = K3 in {32, 64, 128} at 2, 64 at 4, others keep one CTA). Process-wide, default 1; affects launches
// issued afterwards. Returns -1 for other values. Results are bitwise the same for every value.
int set_slab_split(int fwd_ctas, int inv_ctas);
int slab_split(int inverse);

// Raise the dynamic shared-memory limit of the large-footprint kernels (once per device).
cudaError_t configure_kernels();
// Load the kernels that need no such limit (a kernel is loaded when it is first named to the runtime).
cudaError_t load_stage_kernels();
inline cudaError_t set_dynamic_smem(const void *fn, size_t bytes) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

using StageKernel = void (*)(SysDev);
// The slab and influence kernels for a system's plans (fwd.cu, conv.cu, inv.cu); configure_transforms raises the
// shared-memory limits of the three (a plan does it when it is created, which loads only the kernels in use).
StageKernel fwd_kernel(const SysDev &d);
StageKernel conv_kernel(const SysDev &d);
StageKernel inv_kernel(const SysDev &d);
cudaError_t configure_transforms(const SysDev &d);

// Optional device-to-device copies of intermediate meshes (diagnostics).
struct DebugTaps {
    unsigned long long *mesh_out;  // fixed-point charge mesh after spreading, K1*K2*K3
    float *phi_out;                // potential mesh after the inverse FFT, K1*K2*K3
};

enum Stage { STAGE_BIN = 0, STAGE_SPREAD, STAGE_FWD, STAGE_CONV, STAGE_INV, STAGE_GATHER, NUM_STAGES };

// Enqueue the copy of nf floats from device memory to page-locked host memory (dst: its device-side
// address), of the control block ctl to its host copy hctl (device-side address; may be null) and, when
// res8 (device-side address of page-locked memory) is given, of energy, virial and status bits to res8[0..7],
// after the work before it on s.
cudaError_t launch_copy_out(const float *src, float *dst, long long nf, const Ctl *ctl, Ctl *hctl, cudaStream_t s,
                            double *res8 = nullptr);

// Enqueue one stage kernel of system d.
void launch_stage(const SysDev &d, int stage, cudaStream_t s);
// The forward, influence or inverse stage over its work items [first, first + count) only (a rank's planes or
// columns in the slab decomposition).
void launch_stage_items(const SysDev &d, int stage, int first, int count, cudaStream_t s);

// Tensor-core influence stage (tc_dft.cu): kernel set-up, tiles per evaluation, launch, and the DFT-matrix
// image (three BF16 terms of the real and imaginary parts, both K halves, 128-byte swizzled K-major rows).
cudaError_t configure_tc_kernel();
int tc_tiles(const SysDev &d);
cudaError_t launch_conv_tc(const SysDev &d, const void *w_img, cudaStream_t s);
void make_tc_w_image(std::vector<uint8_t> &img);
constexpr size_t TC_W_IMAGE_BYTES = 2 * 6 * 128 * 128;

// Enqueue the six stage kernels of one evaluation of system d on stream s.
cudaError_t launch_pipeline(const SysDev &d, cudaStream_t s, const DebugTaps *taps = nullptr);

}  // namespace pme
