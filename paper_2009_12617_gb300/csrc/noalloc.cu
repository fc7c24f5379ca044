// Allocation-free single-system evaluation: pme_compute_noalloc.
//
// Who needs it: callers that must not allocate device memory themselves. An application that has
// handed all device memory to its own pool up front (a caching allocator, an arena sized at start-up)
// may have nothing left for cudaMalloc, and cudaMalloc / cudaFree synchronise the device, which a
// latency-bound caller (a request loop, a real-time controller) cannot afford on every call. Such
// callers pass only their inputs and outputs; everything else lives in a fixed static device array.
//
// How: a set-up kernel clears what must start at zero and writes the mesh's tables, then the six stage kernels of
// an ordinary evaluation follow on the stream, the last of them storing the result in page-locked host memory. All
// scratch is carved out of g_noalloc_scratch, a file-scope static __device__ array of NOALLOC_SCRATCH_BYTES that every GPU
// loading the library holds until exit. Every kernel a call may need is loaded by the first call on a device
// (loading one later could take device memory).
//
// 2048 atoms, 32^3, p = 4: 52 to 57 us a call. One cooperative kernel with nine grid barriers, its table from
// a division and two exponentials more per point and its transforms in shared memory took 97 us (88 on the GPU).
#include <cuda_runtime.h>
#include <string.h>

#include <mutex>

#include "../../include/pme.h"
#include "host_tables.h"
#include "kernels.h"
#include "pdl.cuh"
#include "plan_internal.h"

namespace pme {

constexpr size_t NOALLOC_SCRATCH_BYTES = (size_t)4 << 20;  // 4 MiB per device
constexpr int NOALLOC_MAX_MESH_POINTS = 32768;             // K1 * K2 * K3 (e.g. 32^3)
constexpr int64_t NOALLOC_MAX_ATOMS = 16384;
constexpr int NOALLOC_THREADS = 128;
constexpr int NOALLOC_MAX_EDGE = 64;

}  // namespace pme

// The scratch array. In host code this name is only a stand-in for the device symbol; its device address
// comes from cudaGetSymbolAddress in noalloc_setup().
static __device__ __align__(256) unsigned char g_noalloc_scratch[pme::NOALLOC_SCRATCH_BYTES];

namespace pme {

struct NoallocArgs {
    int K1, K2, K3, H3;
    double g[6];      // |m'|^2 = g0 m1^2 + g1 m2^2 + g2 m3^2 + g3 m1 m2 + g4 m1 m3 + g5 m2 m3
    double fac;       // pi^2 / beta^2
    double inv_piv;   // 1 / (pi V)
    float4 *bc;       // influence table (SysDev::bc)
    float2 *tw;       // twiddles: K1, K2, K3/2, K3/2 + 1 entries (SysDev::tw1, tw2, tw3h, tw3)
    unsigned long long *zero;  // what must be zero before binning
    int nzero;                 // 8-byte words
};

// M_P(x) at the integer x, by the recursion over orders.
template <int P>
__host__ __device__ constexpr double spline_knot(int x) {
    if constexpr (P == 2) {
        return x == 1 ? 1.0 : 0.0;
    } else {
        return ((double)x * spline_knot<P - 1>(x) + (double)(P - x) * (x >= 1 ? spline_knot<P - 1>(x - 1) : 0.0)) / (P - 1);
    }
}

__device__ __forceinline__ int dev_signed_freq(int m, int K) { return 2 * m <= K ? m : m - K; }

__device__ __forceinline__ double dev_norm2(const NoallocArgs &A, int mt1, int mt2, int mt3) {
    const double x = mt1, y = mt2, z = mt3;
    return fma(x, fma(A.g[0], x, fma(A.g[3], y, A.g[4] * z)), fma(y, fma(A.g[1], y, A.g[5] * z), A.g[2] * z * z));
}

// Clears the charge mesh, counters, partials and control block, and writes the twiddles and the influence table,
// all in FP64 rounded once. Each block keeps B's factors of the three axes in shared memory: with the knots
// symmetric about P / 2, |sum_k M_P(k + 1) exp(2 pi i m k / K)| = |M_P(P/2) + 2 sum_d M_P(P/2 + d) cos(2 pi m d / K)|.
// The FP64 pipe (1/64 of FP32: a warp's instruction holds it for 64 cycles) bounds this kernel, so what counts is the
// number of FP64 instructions in a row of one warp per scheduler: 128 threads a block and a point a thread at 32^3
// (256 threads left half the blocks without points, 13.9 -> 7.9 us), one exponential and one division a point, and
// as much again on Nyquist planes; the last block, which has the fewest points, takes the twiddles.
template <int P>
__global__ void __launch_bounds__(NOALLOC_THREADS) k_noalloc_setup(NoallocArgs A) {
    __shared__ double bm[3 * NOALLOC_MAX_EDGE];
    pdl_wait();
    const int tid = threadIdx.x, nth = blockDim.x, gtid = blockIdx.x * nth + tid, gnth = gridDim.x * nth;
    for (int i = gtid; i < A.nzero; i += gnth) A.zero[i] = 0ull;
    const int K1 = A.K1, K2 = A.K2, K3 = A.K3, H3 = A.H3, Nh = K3 / 2;
    constexpr double knots[4] = {spline_knot<P>(P / 2), spline_knot<P>(P / 2 + 1), spline_knot<P>(P / 2 + 2), spline_knot<P>(P / 2 + 3)};
    for (int i = tid; i < K1 + K2 + H3; i += nth) {
        const int al = i < K1 ? 0 : (i < K1 + K2 ? 1 : 2), m = i - (al == 0 ? 0 : (al == 1 ? K1 : K1 + K2));
        const int K = al == 0 ? K1 : (al == 1 ? K2 : K3);
        double s = knots[0];
#pragma unroll
        for (int k = 1; k < P / 2; ++k) s += 2.0 * knots[k] * cospi((double)(2 * ((m * k) % K)) / (double)K);
        bm[al * NOALLOC_MAX_EDGE + m] = 1.0 / (s * s);
    }
    if (blockIdx.x == gridDim.x - 1)
        for (int i = tid; i < K1 + K2 + Nh + Nh + 1; i += nth) {
            int k = i, len = K1;
            if (k >= K1) {
                k -= K1, len = K2;
                if (k >= K2) {
                    k -= K2, len = Nh;
                    if (k >= Nh) k -= Nh, len = K3;
                }
            }
            double s, c;
            sincospi(-2.0 * (double)k / (double)len, &s, &c);
            A.tw[i] = make_float2((float)c, (float)s);
        }
    __syncthreads();
    // on the half spectrum, [m2][m1][m3]: B(m) (C(m) + C(-m)) / 2 as (hi, lo) floats, then B C f(m) and, off the
    // self-conjugate planes on a Nyquist plane, B C f(m_p), f = 2 (1 / |m'|^2 + pi^2 / beta^2)
    for (int i = gtid; i < K1 * K2 * H3; i += gnth) {
        const int m3 = i % H3, m1 = (i / H3) % K1, m2 = i / (H3 * K1);
        double v = 0.0, g = 0.0, gp = 0.0;
        if (m1 | m2 | m3) {
            const int mt1 = dev_signed_freq(m1, K1), mt2 = dev_signed_freq(m2, K2);
            const double B = bm[m1] * bm[NOALLOC_MAX_EDGE + m2] * bm[2 * NOALLOC_MAX_EDGE + m3] * A.inv_piv;
            const double nm = dev_norm2(A, mt1, mt2, m3), inv = 1.0 / nm;
            v = exp(-A.fac * nm) * inv;
            if (2 * m1 == K1 || 2 * m2 == K2 || 2 * m3 == K3) {
                // the index of -m keeps the frequency +K/2 on a Nyquist axis
                const int p1 = 2 * m1 == K1 ? mt1 : -mt1, p2 = 2 * m2 == K2 ? mt2 : -mt2;
                const double np = dev_norm2(A, p1, p2, 2 * m3 == K3 ? m3 : -m3), inp = 1.0 / np;
                v = 0.5 * (v + exp(-A.fac * np) * inp);
                const bool self = m3 == 0 || 2 * m3 == K3;
                if (!self && (2 * m1 == K1 || 2 * m2 == K2)) gp = v * B * 2.0 * (inp + A.fac);
            }
            v *= B;
            g = v * 2.0 * (inv + A.fac);
        }
        const float hi = (float)v;
        A.bc[i] = make_float4(hi, (float)(v - (double)hi), (float)g, (float)gp);
    }
}

struct NoallocDevice {
    bool ready = false;
    unsigned char *scratch = nullptr;  // device address of g_noalloc_scratch
    int sms = 0;
    double *result = nullptr, *result_dev = nullptr;  // page-locked result (8 doubles) and its device address
};

static std::mutex g_noalloc_mu;
static NoallocDevice g_noalloc_dev[64];

static const void *setup_kernel(int p) {
    return p == 4 ? (const void *)k_noalloc_setup<4> : (p == 6 ? (const void *)k_noalloc_setup<6> : (const void *)k_noalloc_setup<8>);
}

// Once per device, with that device current: the scratch array's device address, the page-locked result block, and
// every kernel that a later call may launch loaded.
static pme_status noalloc_setup(int dev, NoallocDevice **out) {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (dev < 0 || dev >= 64) return fail(PME_ECUDA, "device index %d out of range", dev);
    NoallocDevice &nd = g_noalloc_dev[dev];
    if (!nd.ready) {
        void *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        if ((e = cudaDeviceGetAttribute(&nd.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
            return cuda_fail(e, "cudaDeviceGetAttribute");
        if ((e = ensure_configured(dev)) != cudaSuccess) return cuda_fail(e, "configure kernels");
        cudaFuncAttributes fa;
        for (int p : {4, 6, 8})
            if ((e = cudaFuncGetAttributes(&fa, setup_kernel(p))) != cudaSuccess) return cuda_fail(e, "cudaFuncGetAttributes");
        if ((e = load_stage_kernels()) != cudaSuccess) return cuda_fail(e, "cudaFuncGetAttributes");
        // the transforms of every accepted mesh: influence kernels go by K1, slab kernels by K2 and K3 (with those of the
        // cubic meshes alone, the first call took 32.3 instead of 33.5 ms and later ones 4 MiB of device memory)
        const double recip[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};
        const int smallest = mesh_edge(0);
        auto load = [&](int K1, int K2, int K3) -> cudaError_t {
            const int K[3] = {K1, K2, K3};
            SysDev d;
            memset(&d, 0, sizeof(d));
            fill_geometry(d, K, 4, 1.0, recip);
            return configure_transforms(d);
        };
        for (int i = 0; i < N_EDGES && mesh_edge(i) <= NOALLOC_MAX_EDGE; ++i) {
            if ((e = load(mesh_edge(i), smallest, smallest)) != cudaSuccess) return cuda_fail(e, "configure kernels");
            for (int j = 0; j < N_EDGES && mesh_edge(j) <= NOALLOC_MAX_EDGE; ++j)
                if (smallest * mesh_edge(i) * mesh_edge(j) <= NOALLOC_MAX_MESH_POINTS &&
                    (e = load(smallest, mesh_edge(i), mesh_edge(j))) != cudaSuccess)
                    return cuda_fail(e, "configure kernels");
        }
        if (!nd.result && (e = lib_malloc_host((void **)&nd.result, 8 * sizeof(double))) != cudaSuccess) {
            nd.result = nullptr;
            return cuda_fail(e, "cudaMallocHost");
        }
        if ((e = cudaHostGetDevicePointer((void **)&nd.result_dev, nd.result, 0)) != cudaSuccess)
            return cuda_fail(e, "cudaHostGetDevicePointer");
        nd.scratch = (unsigned char *)ptr;
        nd.ready = true;
    }
    *out = &nd;
    return PME_OK;
}

static size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace pme

using namespace pme;

extern "C" pme_status pme_compute_noalloc(const int K[3], int p, double beta, const double box[9], const float *pos,
                                          const float *q, int64_t n, float *forces, double *energy, double *virial,
                                          void *cuda_stream) {
    if (!K || !box) return fail(PME_EINVAL, "K and box must be non-NULL");
    char msg[256];
    const int v = validate_params(K, p, beta, box, msg, sizeof(msg));
    if (v == 1) return fail(PME_EINVAL, "%s", msg);
    if (v == 2) return fail(PME_EUNSUPPORTED, "%s", msg);
    if (p != 4 && p != 6 && p != 8) return fail(PME_EUNSUPPORTED, "pme_compute_noalloc: B-spline orders 4, 6 and 8 only");
    const int64_t mesh = (int64_t)K[0] * K[1] * K[2];
    if (mesh > NOALLOC_MAX_MESH_POINTS || K[0] > NOALLOC_MAX_EDGE || K[1] > NOALLOC_MAX_EDGE || K[2] > NOALLOC_MAX_EDGE)
        return fail(PME_EINVAL, "pme_compute_noalloc: mesh %dx%dx%d exceeds its static limit (K1*K2*K3 <= %d, each K <= 64)",
                    K[0], K[1], K[2], NOALLOC_MAX_MESH_POINTS);
    if (n < 0 || n > NOALLOC_MAX_ATOMS)
        return fail(PME_EINVAL, "pme_compute_noalloc: n = %lld outside [0, %lld]", (long long)n, (long long)NOALLOC_MAX_ATOMS);
    if (n > 0 && (!pos || !q || !forces)) return fail(PME_EINVAL, "pos, q and forces must be non-NULL when n > 0");
    double recip[9], vol;
    if (!cell_reciprocal(box, recip, &vol)) return fail(PME_EINVAL, "box is singular");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    NoallocDevice *nd = nullptr;
    pme_status st = noalloc_setup(dev, &nd);
    if (st != PME_OK) return st;

    // carve the static scratch: everything that must start at zero comes first. The space set aside for partials and
    // tables is that of the finest division of the influence stage, CONV_COLS columns of one m2 an item.
    SysDev d;
    memset(&d, 0, sizeof(d));
    fill_geometry(d, K, p, beta, recip);
    const size_t K1 = K[0], K2 = K[1], K3 = K[2], H3 = d.H3, Nh = K3 / 2;
    const size_t par_bytes = (K2 * (size_t)d.nchunk3 + K1) * 8 * sizeof(float2);
    const int64_t ncap = n > 0 ? n : 1;
    const int cap = bucket_capacity(ncap, d);
    size_t off = 0;
    const size_t o_ctl = off;  off = al256(off + sizeof(Ctl));
    const size_t o_cnt = off;  off = al256(off + bcount_bytes(d.ntiles));
    const size_t o_qs = off;   off = al256(off + QABS_BYTES);
    const size_t o_par = off;  off = al256(off + par_bytes);
    const size_t o_grid = off; off = al256(off + K1 * K2 * K3 * 8);
    const size_t zero_bytes = off;
    off = al256(off + (K1 + K2 + K3) * 8);  // unused: the call accepts what it did when B's factors were kept here
    const size_t o_tw = off;   off = al256(off + (K1 + K2 + Nh + Nh + 1) * 8);
    const size_t o_bc = off;   off = al256(off + K1 * K2 * H3 * sizeof(float4));
    const size_t o_spec = off; off = al256(off + K1 * K2 * H3 * 8);
    const size_t o_phi = off;  off = al256(off + K1 * K2 * K3 * 4);
    const size_t o_bka = off;  off = al256(off + (size_t)d.ntiles * cap * 16);
    const size_t o_bkb = off;  off = al256(off + (size_t)d.ntiles * cap * 8);
    const size_t o_ova = off;  off = al256(off + (size_t)ncap * 16);
    const size_t o_ovb = off;  off = al256(off + (size_t)ncap * 8);
    if (off > NOALLOC_SCRATCH_BYTES)
        return fail(PME_EINVAL, "pme_compute_noalloc: this system needs %zu bytes of scratch; the static limit is %zu",
                    off, NOALLOC_SCRATCH_BYTES);
    unsigned char *b = nd->scratch;
    d.ctl = (Ctl *)(b + o_ctl);
    d.bcount = (unsigned *)(b + o_cnt);
    d.qslot = (unsigned long long *)(b + o_qs);
    d.partials = (double *)(b + o_par);
    d.grid = (unsigned long long *)(b + o_grid);
    NoallocArgs A;
    memset(&A, 0, sizeof(A));
    A.tw = (float2 *)(b + o_tw);
    d.tw1 = A.tw;
    d.tw2 = A.tw + K1;
    d.tw3h = A.tw + K1 + K2;
    d.tw3 = A.tw + K1 + K2 + Nh;
    A.bc = (float4 *)(b + o_bc);
    d.bc = A.bc;
    d.spec = (float2 *)(b + o_spec);
    d.phi = (float *)(b + o_phi);
    d.bka = (float4 *)(b + o_bka);
    d.bkb = (int2 *)(b + o_bkb);
    d.ova = (float4 *)(b + o_ova);
    d.ovb = (int2 *)(b + o_ovb);
    d.cap = cap;
    d.n = (int)n;
    d.nbin = (int)((n + BIN_CHUNK - 1) / BIN_CHUNK);
    d.pos = pos;
    d.q = q;
    d.forces = forces;
    d.ev = nd->result_dev;  // the final reduction stores energy, virial and status bits there
    d.ev_status = 1;
    A.K1 = K[0];
    A.K2 = K[1];
    A.K3 = K[2];
    A.H3 = d.H3;
    for (int al = 0; al < 3; ++al)
        for (int be = al; be < 3; ++be) {
            double dot = 0.0;
            for (int j = 0; j < 3; ++j) dot += recip[3 * al + j] * recip[3 * be + j];
            A.g[al == be ? al : (al == 0 ? 2 + be : 5)] = al == be ? dot : 2.0 * dot;
        }
    A.fac = PI_D * PI_D / (beta * beta);
    A.inv_piv = 1.0 / (PI_D * vol);
    A.zero = (unsigned long long *)b;
    A.nzero = (int)(zero_bytes / 8);

    cudaStream_t stream = (cudaStream_t)cuda_stream;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nd->sms);
    cfg.blockDim = dim3(NOALLOC_THREADS);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = launch_mode() ? 1 : 0;
    void *args[] = {&A};
    if ((e = cudaLaunchKernelExC(&cfg, setup_kernel(p), args)) != cudaSuccess) return cuda_fail(e, "kernel launch");
    if ((e = launch_pipeline(d, stream)) != cudaSuccess) return cuda_fail(e, "kernel launch");
    if ((e = cudaStreamSynchronize(stream)) != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    const double *r = nd->result;
    if ((st = status_from_bits((unsigned)r[7])) != PME_OK) return st;
    if (energy) *energy = r[0];
    if (virial)
        for (int c = 0; c < 6; ++c) virial[c] = r[1 + c];
    return PME_OK;
}
