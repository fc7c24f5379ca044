// Lane plans of the register transforms and the launch rules that go by them, compiled for the CPU (tests only).
#define PME_HOST_EMULATION 1
#include <stdint.h>
#include <string.h>

#include "../../paper_2009_12617_gb300/csrc/host_tables.h"
#include "../../paper_2009_12617_gb300/csrc/kernels.h"

using namespace pme;

extern "C" {

int lane_edges(int *out) {
    for (int i = 0; i < N_EDGES; ++i) out[i] = mesh_edge(i);
    return N_EDGES;
}

// Threads of the slab CTAs of K2 x K3 slabs: of a single system (slabs 0), or of a group with that many.
int lane_slab_threads(int K2, int K3, int slabs) {
    const int pr = slab_lane_plan(K3 / 2, K2), pc = slab_lane_plan(K2, K3 / 2 + 1);
    return slabs ? slab_group_nt(pr, pc, slabs) : slab_nt(pr, pc);
}

// Default tile edge for n atoms on a GPU with 152 SMs.
int lane_tile_edge(long long n, const int *K, int p) { return 1 << choose_tile_log(n, K, GB300_SMS, p); }

// Bucket capacity for n atoms with tiles of an edge, in as many k1 pieces as a single system has.
int lane_bucket_capacity(long long n, const int *K, int edge) {
    SysDev d;
    memset(&d, 0, sizeof(d));
    d.K1 = K[0];
    d.K2 = K[1];
    d.K3 = K[2];
    d.p = 4;
    set_tiling(d, edge == 16 ? 4 : 3);
    set_tiling(d, d.tlog, choose_k1_pieces(d, GB300_SMS));
    return bucket_capacity(n, d);
}

}  // extern "C"
