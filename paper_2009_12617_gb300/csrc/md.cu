// Device-resident multi-step loop: M time steps of (reciprocal-space SPME forces [+ real-space forces] ->
// leapfrog update of velocities and positions) with no host round trip between steps, the way the paper's
// long-range pipeline runs "multiple timesteps" on its FPGAs without host communication beyond
// initialization and result collection (Sec. III). One chunk of steps is recorded once as a CUDA graph and
// replayed; a device-side step counter tells each step's update kernel where to store that step's energies,
// so every chunk replays the same graph.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "../../include/pme.h"
#include "kernels.h"
#include "plan_internal.h"

namespace pme {

constexpr int MD_CHUNK = 32;   // steps per recorded graph
constexpr int MD_EV = 15;      // doubles per step in ev_steps: E_rec, virial_rec[6], E_real, E_self, virial_real[6]
constexpr size_t MD_MEM = 256; // step counters of the update and of the real-space energies, 128 bytes apart

struct LeapArgs {
    float *pos, *vel, *forces;  // forces: the reciprocal part, replaced by the sum where there is a real part
    const float *real, *inv_mass;  // real-space part or null; null: unit mass
    int n;
    float dt;
    const double *ev_rec;   // the plan's energy / virial of this step (7 doubles)
    double *ev_steps;       // steps x MD_EV or null (the real-space columns are filed by its own reduction)
    unsigned *counter;      // steps completed in this call
    int steps;
};

// v += (F / m) dt, x += v dt, each product and sum rounded once in FP32 (so a host loop of the same
// operations reproduces the trajectory bit for bit); block 0 files the step's energies and advances the
// step counter.
__global__ void __launch_bounds__(256) k_leapfrog(LeapArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.n) {
        const float im = a.inv_mass ? a.inv_mass[i] : 1.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const size_t j = 3 * (size_t)i + k;
            float f = a.forces[j];
            if (a.real) {
                f = __fadd_rn(f, a.real[j]);
                a.forces[j] = f;
            }
            const float v = __fadd_rn(a.vel[j], __fmul_rn(__fmul_rn(f, im), a.dt));
            a.vel[j] = v;
            a.pos[j] = __fadd_rn(a.pos[j], __fmul_rn(v, a.dt));
        }
    }
    if (blockIdx.x == 0) {
        __shared__ unsigned step;
        if (threadIdx.x == 0) step = *a.counter;
        __syncthreads();
        if (a.ev_steps && step < (unsigned)a.steps && threadIdx.x < (a.real ? 7 : MD_EV)) {
            const int t = threadIdx.x;
            a.ev_steps[(size_t)step * MD_EV + t] = t < 7 ? a.ev_rec[t] : 0.0;
        }
        __syncthreads();
        if (threadIdx.x == 0) *a.counter = step + 1u;
    }
}

static cudaError_t launch_leapfrog(const LeapArgs &a, cudaStream_t s) {
    const unsigned g = (unsigned)(a.n > 0 ? (a.n + 255) / 256 : 1);
    k_leapfrog<<<g, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace pme

using namespace pme;

extern "C" pme_status pme_run_steps(pme_plan *pl, pme_real *rs, float *pos, float *vel, const float *q,
                                    const float *inv_mass, int64_t n, float *forces, double dt, int steps,
                                    double *ev_steps) {
    pme_status st = check_atoms(pl, pos, q, n, forces);
    if (st) return st;
    if (n > 0 && !vel) return fail(PME_EINVAL, "vel must be non-NULL when n > 0");
    if (steps < 0 || !(dt == dt) || !isfinite(dt)) return fail(PME_EINVAL, "steps must be >= 0 and dt finite");
    if (rs && real_device(rs) != pl->dev) return fail(PME_EINVAL, "the real-space context lives on another device");
    DeviceGuard g(pl->dev);
    if ((st = plan_reserve(pl, n)) != PME_OK) return st;
    if (rs && (st = real_reserve_n(rs, n)) != PME_OK) return st;
    cudaError_t e;
    if (!pl->md_mem) {
        if ((e = lib_malloc(&pl->md_mem, MD_MEM)) != cudaSuccess) {
            pl->md_mem = nullptr;
            return fail(PME_ENOMEM, "cudaMalloc(step-loop state): %s", cudaGetErrorString(e));
        }
    }
    if (steps == 0) return PME_OK;
    unsigned *counter = (unsigned *)pl->md_mem, *real_counter = counter + 32;
    if ((e = cudaMemsetAsync(pl->md_mem, 0, MD_MEM, pl->stream)) != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
    if (rs && !pl->md_done) {
        int least = 0, greatest = 0;
        if ((e = cudaDeviceGetStreamPriorityRange(&least, &greatest)) != cudaSuccess) return cuda_fail(e, "stream priorities");
        if ((!pl->md_main && (e = cudaStreamCreateWithPriority(&pl->md_main, cudaStreamNonBlocking, greatest)) != cudaSuccess) ||
            (!pl->md_side && (e = cudaStreamCreateWithPriority(&pl->md_side, cudaStreamNonBlocking, least)) != cudaSuccess))
            return cuda_fail(e, "cudaStreamCreate");
        for (cudaEvent_t *ev : {&pl->md_fork, &pl->md_pairs, &pl->md_done})
            if (!*ev && (e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) {
                *ev = nullptr;
                return cuda_fail(e, "cudaEventCreate");
            }
    }

    const SysDev d = plan_descriptor(pl, pos, q, n, forces, nullptr);
    LeapArgs la;
    la.pos = pos;
    la.vel = vel;
    la.forces = forces;
    la.real = nullptr;
    la.inv_mass = inv_mass;
    la.n = (int)n;
    la.dt = (float)dt;
    la.ev_rec = pl->d.ctl->ev;
    la.ev_steps = ev_steps;
    la.counter = counter;
    la.steps = steps;
    // One step on stream s: reciprocal forces, then the update. With real space, its kernels run beside the
    // reciprocal stages on the side stream into an array of their own, and the update adds the two parts (the same
    // sums as one after the other); the real-space energies are reduced beside the update. The stages leave most
    // of the GPU idle (six latency chains), and the pair kernel fills it: 8190 atoms, 40^3, 63 -> 38 us a step.
    auto one_step = [&](cudaStream_t s) -> cudaError_t {
        cudaError_t r;
        if (rs) {
            if ((r = cudaEventRecord(pl->md_fork, s)) != cudaSuccess || (r = cudaStreamWaitEvent(pl->md_side, pl->md_fork, 0)) != cudaSuccess)
                return r;
            la.real = real_enqueue_own(rs, pl->md_side, pos, q, n);
            if ((r = cudaEventRecord(pl->md_pairs, pl->md_side)) != cudaSuccess) return r;
            real_enqueue_file(rs, pl->md_side, n, real_counter, ev_steps ? ev_steps + 7 : nullptr, MD_EV, steps);
        }
        if ((r = launch_pipeline(d, s)) != cudaSuccess) return r;
        if (rs && (r = cudaStreamWaitEvent(s, pl->md_pairs, 0)) != cudaSuccess) return r;
        return launch_leapfrog(la, s);
    };
    // the side stream's last work back into s
    auto join = [&](cudaStream_t s) -> cudaError_t {
        if (!rs) return cudaSuccess;
        const cudaError_t r = cudaEventRecord(pl->md_done, pl->md_side);
        return r != cudaSuccess ? r : cudaStreamWaitEvent(s, pl->md_done, 0);
    };
    const int chunk = steps < MD_CHUNK ? steps : MD_CHUNK;
    pme_plan::StepGraph key;
    key.pos = pos;
    key.vel = vel;
    key.q = q;
    key.inv_mass = inv_mass;
    key.forces = forces;
    key.ev_steps = ev_steps;
    key.rs = rs;
    key.atoms = pl->atom_mem;
    key.n = n;
    key.chunk = chunk;
    key.mode = launch_mode();
    key.dt = dt;
    key.gen = pl->gen;
    key.rs_gen = rs ? real_gen(rs) : 0ull;
    pme_plan::StepGraph &gm = pl->g_md;
    const bool same = gm.exec && gm.pos == key.pos && gm.vel == key.vel && gm.q == key.q && gm.inv_mass == key.inv_mass &&
                      gm.forces == key.forces && gm.ev_steps == key.ev_steps && gm.rs == key.rs && gm.atoms == key.atoms &&
                      gm.n == key.n && gm.chunk == key.chunk && gm.mode == key.mode && gm.dt == key.dt && gm.gen == key.gen &&
                      gm.rs_gen == key.rs_gen;
    if (!same) {
        if (gm.exec) cudaGraphExecDestroy(gm.exec);
        gm = pme_plan::StepGraph();
        if (!pl->rec_stream && (e = cudaStreamCreateWithFlags(&pl->rec_stream, cudaStreamNonBlocking)) != cudaSuccess)
            return cuda_fail(e, "cudaStreamCreate");
        const cudaStream_t rec = rs ? pl->md_main : pl->rec_stream;
        if ((e = cudaStreamBeginCapture(rec, cudaStreamCaptureModeThreadLocal)) != cudaSuccess)
            return cuda_fail(e, "cudaStreamBeginCapture");
        cudaError_t r = cudaSuccess;
        for (int i = 0; i < chunk && r == cudaSuccess; ++i) r = one_step(rec);
        if (r == cudaSuccess) r = join(rec);
        cudaGraph_t graph = nullptr;
        e = cudaStreamEndCapture(rec, &graph);
        if (r != cudaSuccess || e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            return cuda_fail(r != cudaSuccess ? r : e, "recording the step loop");
        }
        cudaGraphExec_t exec = nullptr;
        e = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate(step loop)");
        gm = key;
        gm.exec = exec;
    }
    for (int done = 0; done + chunk <= steps; done += chunk)
        if ((e = cudaGraphLaunch(gm.exec, pl->stream)) != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch(step loop)");
    for (int i = steps - steps % chunk; i < steps; ++i)  // the remainder, launched directly
        if ((e = one_step(pl->stream)) != cudaSuccess) return cuda_fail(e, "step launch");
    if (steps % chunk && (e = join(pl->stream)) != cudaSuccess) return cuda_fail(e, "step launch");
    return PME_OK;
}
