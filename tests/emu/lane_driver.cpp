// The register transforms, run by a warp of 32 CPU threads, and the launch rules of the stages (tests only).
#define PME_HOST_EMULATION 1
#define PME_EMULATE_WARP 1
#include <sched.h>
#include <stdint.h>
#include <string.h>

#include <atomic>
#include <limits>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

// the warp: lanes meet at a barrier before and after every exchange
static thread_local struct {
    unsigned x;
} threadIdx;
static float g_word[32];
static std::atomic<unsigned> g_arrived, g_round;
static void warp_barrier() {
    const unsigned r = g_round.load();
    if (g_arrived.fetch_add(1) == 31) {
        g_arrived.store(0);
        g_round.store(r + 1);
    } else {
        while (g_round.load() == r) sched_yield();
    }
}
static float __shfl_sync(unsigned, float v, int lane) {
    g_word[threadIdx.x] = v;
    warp_barrier();
    const float r = g_word[lane & 31];
    warp_barrier();
    return r;
}
static float __shfl_xor_sync(unsigned m, float v, int mask) { return __shfl_sync(m, v, (int)threadIdx.x ^ mask); }
template <class T>
static T __ldg(const T *p) {
    return *p;
}

#include "../../paper_2009_12617_gb300/csrc/host_tables.h"
#include "../../paper_2009_12617_gb300/csrc/kernels.h"
#include "../../paper_2009_12617_gb300/csrc/stages.cuh"

using namespace pme;

// One lane's part of the transforms of a plan: in holds T transforms of N points; fwd and inv get them transformed
// either way, back the adjoint of the forward transform applied to it. Stores as the slab and influence stages do.
template <int L, int E>
static void lane_transforms(const float2 *in, const float2 *twiddles, float2 *fwd, float2 *inv, float2 *back) {
    constexpr int N = L * E, T = 32 / L;
    int t, j;
    lane_unit<L>((int)threadIdx.x, t, j);
    const bool ok = t < T;
    const int tt = ok ? t : 0, r = lane_rev<L>(j);
    const LaneTw<L, E> tw = lane_tw<L, E, true>(twiddles, j);
    float2 v[E], w[E];
    for (int n = 0; n < E; ++n) v[n] = w[n] = in[tt * N + j + L * n];
    lane_fft<L, E, false>(v, j, tw);
    lane_fft<L, E, true>(w, j, tw);
    if (ok)
        for (int k = 0; k < E; ++k) {
            fwd[t * N + k + E * r] = v[k];
            inv[t * N + k + E * r] = w[k];
        }
    lane_fft_adjoint<L, E>(v, j, tw);
    if (ok)
        for (int n = 0; n < E; ++n) back[t * N + j + L * n] = v[n];
}

extern "C" {

int lane_plans() { return LANE_PLANS; }
void lane_plan(int c, int *out) {
    out[0] = plan_L(c);
    out[1] = plan_E(c);
}

// The transforms of plan c on 32 / L rows of L E complex values. The twiddles lie between NaNs, so that a wrong index
// shows in the results.
void lane_run(int c, const float *in, float *fwd, float *inv, float *back) {
    const int N = plan_L(c) * plan_E(c);
    const float nan = std::numeric_limits<float>::quiet_NaN();
    std::vector<float2> tw(3 * N, make_float2(nan, nan));
    make_twiddles(N, N, tw.data() + N);
    auto lane = [&](int l) {
        threadIdx.x = (unsigned)l;
        switch (c) {
#define PME_RUN(c_, L, E) \
    case c_: lane_transforms<L, E>((const float2 *)in, tw.data() + N, (float2 *)fwd, (float2 *)inv, (float2 *)back); break;
            PME_LANE_CASES(PME_RUN)
#undef PME_RUN
        }
    };
    std::vector<std::thread> warp;
    for (int l = 0; l < 32; ++l) warp.emplace_back(lane, l);
    for (std::thread &t : warp) t.join();
}

// Bytes that the stages of a mesh use of the shared memory they are given, and those: forward, inverse, influence.
void lane_smem(int K1, int K2, int K3, long long *used, long long *given) {
    SysDev d;
    memset(&d, 0, sizeof(d));
    d.K1 = K1;
    d.K2 = K2;
    d.K3 = K3;
    d.H3 = K3 / 2 + 1;
    choose_fft_paths(d, true);
    used[0] = ((long long)K2 * d.zs + K3 / 2 + 1 + K2) * (long long)sizeof(float2);
    used[1] = ((long long)K2 * d.ys + K3 / 2 + K3 / 2 + 1) * (long long)sizeof(float2);
    used[2] = 7ll * CONV_UNITS * (long long)sizeof(float);
    if (d.zs < K3 / 2 || d.ys < d.H3) used[0] = used[1] = 1ll << 40;
    given[0] = (long long)smem_slab(K2, K3);
    given[1] = (long long)smem_inv(K2, K3);
    given[2] = (long long)smem_conv(K1, NT_CONV);
}

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
