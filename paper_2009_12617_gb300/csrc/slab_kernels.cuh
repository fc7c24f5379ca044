// The slab stage kernels, for one system and for a group of systems (batches, server waves). A kernel holds one
// pair of lane plans, fixed at compile time (small enough for the instruction caches): one for every K2 from 16 and
// every K3 within SLAB_NEAR edges of it (of the list of mesh edges), in groups for K2 = K3; other meshes run kernels
// that pick the plans at run time. Included by the files that instantiate the forward and the inverse stage, each
// for every second K2.
//
// A specialised pair saves about 2.4 us of an evaluation over the run-time choice (60^3: 28.5 -> 26.1 us).
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "group.h"
#include "kernels.h"
#include "pdl.cuh"
#include "stages.cuh"

namespace pme {

constexpr int SLAB_NEAR = 3, SLAB_WIDE = 2 * SLAB_NEAR + 1;
constexpr int SLAB_FIRST = 3;  // mesh_edge(3) = 16

// Lane plans of the slabs of K2 = mesh_edge(I), K3 = mesh_edge(J).
template <int I, int J>
struct SlabPlans {
    static constexpr int PR = slab_lane_plan(mesh_edge(J) / 2, mesh_edge(I));
    static constexpr int PC = slab_lane_plan(mesh_edge(I), mesh_edge(J) / 2 + 1);
    static_assert(PR >= 0 && PC >= 0, "every edge has lane plans");
};

// Launch bound of the kernel of a pair of plans.
constexpr int slab_bound(int pr, int pc) { return pr == PLAN_ANY ? NT_SLAB : (pr == PLAN_POW2 ? SLAB_THREADS : slab_nt(pr, pc)); }

// Of the kernels that pick the plans at run time, the one with the power-of-two plans inlined serves the meshes that it
// can: the calls of the other cost them about 1 us of an evaluation (48 x 24 x 96 23.3 -> 22.4 us, 128 x 8 x 128
// 25.4 -> 22.9, 32 x 32 x 64 22.0 -> 20.8, 12^3 18.7 -> 17.3; 16 x 128 x 16 alone gains from them, 21.7 -> 22.2).
inline bool slab_pow2(const SysDev &d, unsigned threads) {
    return d.lp_rows < LANE_POW2_PLANS && d.lp_cols < LANE_POW2_PLANS && threads <= (unsigned)SLAB_THREADS;
}

// Stage is a class with static device functions run<PR, PC>(d, item, smem).
template <class Stage, int PR, int PC>
__global__ void __launch_bounds__(slab_bound(PR, PC)) k_slab(SysDev d) {
    extern __shared__ __align__(16) unsigned char smem[];
    PdlScope pdl(d.pdl_late);
    Stage::template run<PR, PC>(d, d.item0 + blockIdx.x, smem);
}
template <class Stage, int PR, int PC>
__global__ void __launch_bounds__(slab_bound(PR, PC)) k_slab_g(GroupArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SysDev sd;
    PdlScope pdl(a.late);
    const int item = group_load(a, sd);
    Stage::template run<PR, PC>(sd, item, smem);
}

// The kernels for K2 = mesh_edge(I), I = PART, PART + 2, ...; null where there is none.
template <class Stage, int PART>
struct SlabTable {
    static constexpr int ROWS = N_EDGES / 2;
    StageKernel one[ROWS][SLAB_WIDE];
    GroupKernel group[ROWS];

    template <int R, int D>
    static StageKernel pick() {
        constexpr int I = 2 * R + PART, J = I + D - SLAB_NEAR;
        if constexpr (I >= SLAB_FIRST && J >= SLAB_FIRST && J < N_EDGES) return k_slab<Stage, SlabPlans<I, J>::PR, SlabPlans<I, J>::PC>;
        else return nullptr;
    }
    template <int R>
    static GroupKernel pick_group() {
        constexpr int I = 2 * R + PART;
        if constexpr (I >= SLAB_FIRST) return k_slab_g<Stage, SlabPlans<I, I>::PR, SlabPlans<I, I>::PC>;
        else return nullptr;
    }
    template <int R, int... D>
    void fill_row(std::integer_sequence<int, D...>) {
        ((one[R][D] = pick<R, D>()), ...);
        group[R] = pick_group<R>();
    }
    template <int... R>
    void fill(std::integer_sequence<int, R...>) {
        (fill_row<R>(std::make_integer_sequence<int, SLAB_WIDE>()), ...);
    }
    SlabTable() { fill(std::make_integer_sequence<int, ROWS>()); }

    StageKernel find(int i2, int i3) const {
        const int D = i3 - i2 + SLAB_NEAR;
        return D >= 0 && D < SLAB_WIDE ? one[i2 / 2][D] : nullptr;
    }
    GroupKernel find_group(int i2, int i3) const { return i2 == i3 ? group[i2 / 2] : nullptr; }
    cudaError_t configure_group() const {
        for (GroupKernel k : group)
            if (k) {
                const cudaError_t e = set_dynamic_smem((const void *)k, GROUP_SMEM_BYTES);
                if (e != cudaSuccess) return e;
            }
        return cudaSuccess;
    }
};

}  // namespace pme
