// Real-space and self terms of Ewald electrostatics on the GPU: with the reciprocal-space SPME evaluation
// (the paper's long-range pipeline) they make up the full Ewald sum the paper splits its electrostatics
// into (Sec. II; the short-range part runs on its own pipelines beside the long-range one, Sec. III):
//   E_real = 1/2 sum_{i,j,n}' q_i q_j erfc(beta r) / r   over images with r = |r_i - r_j + n| <= rcut,
//   F_i    = sum_{j,n}' q_i q_j [erfc(beta r) / r + 2 beta / sqrt(pi) exp(-beta^2 r^2)] d / r^2,
//   Pi_ab  = 1/2 sum' s_ij d_a d_b   (s_ij the scalar factor of the force, d = r_i - r_j + n),
//   E_self = -beta / sqrt(pi) sum_i q_i^2.
//
// Design. Positions become 32-bit fixed point, modulo 2^32 units u (a power of two chosen so that everything a
// work item looks at lies within 2^31 units): differences of two atoms are exact integer subtractions, images
// are integer offsets, and a displacement is rounded once, when it becomes a float. Cells about half a
// cutoff wide, or a whole one (real_grid; neighbour offsets -R..R), hold the atoms in input-index order, so every sum
// below runs in an order that depends only on the inputs: results are bit-reproducible. A work item is up to 32 consecutive sorted atoms of one row of cells (one lane each) and
// belongs to one CTA, whose warps share out the candidate atoms of the neighbouring rows; see k_rs_pairs. Each
// pair is visited from both ends, so no atom is written by two CTAs and no force atomics are needed. Energies
// are summed per lane in double-float and across work items in FP64 in a fixed order.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>

#include "../../include/pme.h"
#include "common.cuh"
#include "host_tables.h"
#include "kernels.h"
#include "pdl.cuh"
#include "plan_internal.h"

namespace pme {

constexpr int RS_SCAN_THREADS = 1024;
constexpr int RS_BIN_THREADS = 256;
constexpr int RS_RED_BLOCKS = 16;   // level-one blocks of the final reduction
constexpr int RS_MAX_R = 4;         // cutoffs of up to 4 cell widths per axis (cells at least a cutoff wide)
constexpr int RS_MAX_CELLS = 1 << 22;
constexpr int RS_CAND = 192;        // candidates a warp of the pair kernel holds at a time
constexpr int RS_SUMS = 8;          // energy, virial xx yy zz xy xz yz, q^2

struct RealCtl {
    unsigned status;  // StatusBits
    unsigned nitems;  // work items of the pair kernel, written by the scan
    unsigned arrived; // level-one blocks of the reduction that have finished (reset by the last)
    unsigned pad;
    double res[8];    // E_real, E_self, virial xx yy zz xy xz yz
};

// The cells of a box and what goes by them.
struct RealGrid {
    int nc[3], R[3], ncells;
    int slab, nslab, nrowslabs;  // cells along axis 2 per work-item slab, slabs per row, rows x slabs
    float rec[9];          // a*_alpha[j] at 3 alpha + j (cell assignment)
    int afix[9];           // a_alpha[k] / u at 3 alpha + k, low 32 bits of the nearest integer
    float afrac[9];        // what is left of a_alpha[k] / u, in [-1/2, 1/2]
    double inv_u;          // 1 / u
    float inv_u2;          // 1 / u^2
    float rc2, rc2_slack;        // rcut^2 in units^2, and with the candidate test's relative slack
    float beta04_u, ex_k, c2_u;  // 2 beta u / 5; beta^2 u^2 log2(e); 2 beta u / sqrt(pi)
};

struct RealDev : RealGrid {
    int n;
    int max_items;         // launched pair CTAs: n / 32 + one per occupied row slab, at most
    double beta_d;
    int accumulate;        // forces += (1) or = (0)
    const float *pos, *q;
    float *forces;
    double *ev;            // optional device destination of RealCtl::res (8 doubles)
    // optional: step number file_step[0] (advanced here) and a row of file_stride doubles per step, to hold
    // RealCtl::res for steps below file_rows
    unsigned *file_step;
    double *file;
    int file_stride, file_rows;
    RealCtl *host;         // optional page-locked copy of the control block's status and results (device address)
    unsigned *count;       // ncells, zero between calls (reset by the scan)
    unsigned *start;       // ncells + 1
    int2 *cell;            // n: input atom i's cell and arrival number in it
    int4 *xq;              // n: input atom i's fixed-point position in the home cell and charge bits
    int *aidx;             // n: input indices, cell ranges in arrival order
    int4 *sx;              // n: (x, y, z, q bits) in cell order, input order inside a cell
    int *sidx;             // n: input index likewise
    int *scell;            // n: cell likewise
    int2 *items;           // first sorted atom and atom count of each work item
    double *sums;          // RS_SUMS per work item
    float *fown;           // 3 n: forces of real_enqueue_own
    double *partials;      // RS_RED_BLOCKS x 8
    RealCtl *ctl;
};

// fixed-point positions are numbers modulo 2^32
__device__ __forceinline__ int wadd(int a, int b) { return (int)((unsigned)a + (unsigned)b); }
__device__ __forceinline__ int wsub(int a, int b) { return (int)((unsigned)a - (unsigned)b); }
__device__ __forceinline__ int wmul(int a, int b) { return (int)((unsigned)a * (unsigned)b); }
// component k of the cell vector combination m0 a + m1 b + m2 c in units
__device__ __forceinline__ int image_offset(const RealDev &d, int k, int m0, int m1, int m2) {
    const float fr = (float)m0 * d.afrac[k] + (float)m1 * d.afrac[3 + k] + (float)m2 * d.afrac[6 + k];
    return wadd(wadd(wmul(m0, d.afix[k]), wmul(m1, d.afix[3 + k])), wadd(wmul(m2, d.afix[6 + k]), __float2int_rn(fr)));
}

__device__ __forceinline__ int floordiv(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// 1: per atom its cell and arrival number, and its fixed-point position: x / u rounded to an integer (exact
// wherever x's own spacing is at least u), less the whole cells it lies out, both modulo 2^32. An atom without such
// a position (a non-finite coordinate, 2^20 cells out) goes to the origin. It and an atom of non-finite charge carry
// the charge NaN, so that their forces, those around them and the energies show it where nobody asks for the status
// (pme_real_enqueue).
__global__ void __launch_bounds__(RS_BIN_THREADS) k_rs_bin(RealDev d) {
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < d.n) {
        const float r[3] = {d.pos[3 * (size_t)i], d.pos[3 * (size_t)i + 1], d.pos[3 * (size_t)i + 2]};
        const float qq = d.q[i];
        float s[3];
        bool lost = !(isfinite(r[0]) && isfinite(r[1]) && isfinite(r[2]));
#pragma unroll
        for (int al = 0; al < 3; ++al) {
            s[al] = fmaf(r[0], d.rec[3 * al], fmaf(r[1], d.rec[3 * al + 1], r[2] * d.rec[3 * al + 2]));
            if (!(fabsf(s[al]) < 1048576.0f)) lost = true;  // also catches NaN: absurdly far out
        }
        const bool bad = lost || !isfinite(qq);
        if (bad) atomicOr(&d.ctl->status, ST_NONFINITE);
        int c[3] = {0, 0, 0}, X[3] = {0, 0, 0};
        if (!lost) {
            int fl[3];
#pragma unroll
            for (int al = 0; al < 3; ++al) {
                const float w = floorf(s[al]), f = s[al] - w;  // exact: s and floor(s) are within one of each other
                fl[al] = (int)w;
                const int ci = (int)(f * (float)d.nc[al]);
                c[al] = ci < 0 ? 0 : (ci >= d.nc[al] ? d.nc[al] - 1 : ci);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k)
                X[k] = wsub((int)(unsigned)(unsigned long long)__double2ll_rn((double)r[k] * d.inv_u),
                            image_offset(d, k, fl[0], fl[1], fl[2]));
        }
        const int cid = (c[0] * d.nc[1] + c[1]) * d.nc[2] + c[2];
        d.xq[i] = make_int4(X[0], X[1], X[2], bad ? 0x7fc00000 : __float_as_int(qq));
        d.cell[i] = make_int2(cid, (int)atomicAdd(d.count + cid, 1u));
    }
}

// Exclusive scan of one value per thread over the CTA; total receives the sum. Uses warp shuffles and one
// shared word per warp.
__device__ unsigned block_scan(unsigned v, unsigned *wtot, unsigned &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wtot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        unsigned w = lane < nw ? wtot[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        wtot[lane] = w;
    }
    __syncthreads();
    const unsigned before = warp ? wtot[warp - 1] : 0u;
    total = wtot[31];
    __syncthreads();  // wtot may be written again
    return before + x - v;
}

// 2 (one CTA): exclusive scan of the counts into start[], counts reset for the next call, four cells per
// thread and pass; then the work items, one per 32 atoms (or rest) of each row slab, in row-slab order.
__global__ void __launch_bounds__(RS_SCAN_THREADS) k_rs_scan(RealDev d) {
    __shared__ unsigned wtot[32];
    pdl_wait();
    const int t = threadIdx.x;
    unsigned run = 0, total;
    for (int b = 0; b < d.ncells; b += 4 * RS_SCAN_THREADS) {
        const int c = b + 4 * t;
        unsigned k[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            k[j] = c + j < d.ncells ? d.count[c + j] : 0u;
            if (k[j]) d.count[c + j] = 0u;
        }
        unsigned at = run + block_scan(k[0] + k[1] + k[2] + k[3], wtot, total);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (c + j < d.ncells) d.start[c + j] = at;
            at += k[j];
        }
        run += total;
    }
    if (t == 0) d.start[d.ncells] = run;
    __syncthreads();
    run = 0;
    for (int b = 0; b < d.nrowslabs; b += RS_SCAN_THREADS) {
        const int rs = b + t;
        int first = 0, cnt = 0;
        if (rs < d.nrowslabs) {
            const int row = rs / d.nslab, s = rs - row * d.nslab;
            const int z0 = s * d.slab, z1 = min(d.nc[2], z0 + d.slab);
            first = (int)d.start[row * d.nc[2] + z0];
            cnt = (int)d.start[row * d.nc[2] + z1] - first;
        }
        unsigned at = run + block_scan((unsigned)(cnt + 31) >> 5, wtot, total);
        for (int a = 0; a < cnt; a += 32) d.items[at++] = make_int2(first + a, min(32, cnt - a));
        run += total;
    }
    if (t == 0) d.ctl->nitems = run;
}

// 3: input indices into the cells' ranges (arrival order inside a cell).
__global__ void __launch_bounds__(256) k_rs_scatter(RealDev d) {
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= d.n) return;
    const int2 c = d.cell[i];
    d.aidx[d.start[c.x] + (unsigned)c.y] = i;
}

// 4: inside each cell, input-index order: the atom at slot k moves to start + (number of the cell's atoms
// with a smaller input index).
__global__ void __launch_bounds__(256) k_rs_rank(RealDev d) {
    pdl_wait();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n) return;
    const int i = d.aidx[k];
    const int c = d.cell[i].x;
    const unsigned b = d.start[c], e = d.start[c + 1];
    unsigned r = 0;
    for (unsigned j = b; j < e; ++j) r += (unsigned)(d.aidx[j] < i);
    d.sx[b + r] = d.xq[i];
    d.sidx[b + r] = i;
    d.scell[b + r] = c;
}

__device__ __forceinline__ float mufu_rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float mufu_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float mufu_rsqrt(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// exp(x^2) erfc(x) for x >= 0 as t Q(t), t = 1 / (1 + 2 x / 5), Q the degree-10 polynomial that interpolates
// exp(x^2) erfc(x) / t at the Chebyshev nodes of t in (0, 1] (fitted in 40-digit arithmetic; largest relative
// error 1.1e-8, with the coefficients rounded to FP32 2.9e-8, evaluated in FP32 about 2e-7). x04 = 2 x / 5.
__device__ __forceinline__ F2 erfcx_pos(F2 x04) {
    const float2 u = f2_get(f2_add(x04, f2_all(1.0f)));
    const F2 t = f2(mufu_rcp(u.x), mufu_rcp(u.y));
    F2 p = f2_all(-0.0298694347f);
    p = f2_fma(p, t, f2_all(0.143845467f));
    p = f2_fma(p, t, f2_all(-0.243052065f));
    p = f2_fma(p, t, f2_all(0.146816913f));
    p = f2_fma(p, t, f2_all(-0.0538043274f));
    p = f2_fma(p, t, f2_all(0.0871264424f));
    p = f2_fma(p, t, f2_all(0.118093218f));
    p = f2_fma(p, t, f2_all(0.17189095f));
    p = f2_fma(p, t, f2_all(0.207600679f));
    p = f2_fma(p, t, f2_all(0.225676319f));
    p = f2_fma(p, t, f2_all(0.225675831f));
    return f2_mul(p, t);
}

// One neighbouring run of atoms: the part of a row of cells that one image of it contributes.
struct alignas(16) RsPiece {
    int sx, sy, sz;  // fixed-point image offset less the work item's centre
    int first;       // sorted atom first + c is candidate c
};
constexpr int RS_HITS = 96;  // rows of a warp's hit list: 64 and room for one block
struct alignas(16) RsWarp {
    float fx[64], fy[64], fz[64], f2[64];  // candidates not tested yet, a ring: -2 (x, y, z), |x|^2 from the centre
    int4 x[RS_CAND];                       // candidates, a ring: the same in fixed point, and the charge's bits
    unsigned char hit[RS_HITS][32];  // per lane, accepted candidates (ring positions)
};
static_assert(RS_CAND == 192, "six blocks of 32: see rs_block; positions are bytes");
template <int NW>
struct RsShared {
    RsWarp w[NW];
    RsPiece piece[NW * 32];
    int end[NW * 32];  // candidates in pieces 0..p
    int wtot[NW];
};
static_assert(sizeof(RsWarp) >= sizeof(float) * 12 * 32, "the warps' sums are left there");

__device__ __forceinline__ unsigned shared_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// One lane's atom (units relative to the centre), its accepted candidates ("hits"), and its sums: two of each,
// for the first and the second hit of a step.
struct RsLane {
    int x, y, z;
    float q;
    float xf, yf, zf, lim;  // the atom as floats; limit of the candidate test
    unsigned wp, rp, wrap;  // shared addresses of the next hit written and read, and where the reader turns back (0: nowhere)
    int cnt, done;          // hits recorded and evaluated
    unsigned past;          // cnt (mod 256) as it was one to four blocks ago, newest in the low byte
    F2 fx, fy, fz, w[6], eh, el;  // forces, virial; energy as an unevaluated sum
};

// Up to two pending hits of every lane. With r in units: s = q_i q_j exp(-b^2 r^2) (erfcx(b r) + 2 b r /
// sqrt(pi)) / r^3 is the scalar factor of the force, e = q_i q_j exp(-b^2 r^2) erfcx(b r) / r the energy; both
// zero outside the cutoff, for the atom itself and where no hit is pending.
__device__ __forceinline__ void rs_evaluate(const RealDev &d, const RsWarp &W, RsLane &L, unsigned hit0) {
    const int n = L.cnt - L.done;
    int4 J[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        unsigned j;
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(j) : "r"(L.rp));
        J[u] = W.x[n > u ? j : 0u];
        if (n > u) {
            L.rp += 32;
            if (L.rp == L.wrap) {
                L.rp = hit0;
                L.wrap = 0u;
            }
        }
    }
    L.done += min(n, 2);
    const F2 dx = f2((float)(L.x - J[0].x), (float)(L.x - J[1].x)), dy = f2((float)(L.y - J[0].y), (float)(L.y - J[1].y)),
             dz = f2((float)(L.z - J[0].z), (float)(L.z - J[1].z));
    const F2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
    const float2 r2s = f2_get(r2);
    const bool ina = n > 0 && r2s.x <= d.rc2 && r2s.x > 0.f, inb = n > 1 && r2s.y <= d.rc2 && r2s.y > 0.f;
    const float ra = mufu_rsqrt(r2s.x), rb = mufu_rsqrt(r2s.y);
    const F2 rinv = f2(ina ? ra : 0.f, inb ? rb : 0.f);
    const F2 r = f2_mul(r2, rinv);
    const F2 G = erfcx_pos(f2_mul(r, f2_all(d.beta04_u)));
    const float2 ea = f2_get(f2_mul(r2, f2_all(-d.ex_k)));
    const F2 qr = f2_mul(f2_mul(f2_all(L.q), f2(__int_as_float(J[0].w), __int_as_float(J[1].w))), rinv);
    const F2 A = f2_mul(qr, f2(mufu_ex2(ea.x), mufu_ex2(ea.y)));
    const F2 er = f2_mul(A, G);
    const F2 s = f2_mul(f2_mul(A, f2_fma(f2_all(d.c2_u), r, G)), f2_mul(rinv, rinv));
    const F2 sx = f2_mul(s, dx), sy = f2_mul(s, dy), sz = f2_mul(s, dz);
    L.fx = f2_add(L.fx, sx);
    L.fy = f2_add(L.fy, sy);
    L.fz = f2_add(L.fz, sz);
    L.w[0] = f2_fma(sx, dx, L.w[0]);
    L.w[1] = f2_fma(sy, dy, L.w[1]);
    L.w[2] = f2_fma(sz, dz, L.w[2]);
    L.w[3] = f2_fma(sx, dy, L.w[3]);
    L.w[4] = f2_fma(sx, dz, L.w[4]);
    L.w[5] = f2_fma(sy, dz, L.w[5]);
    // two-sum
    const F2 h = f2_add(L.eh, er), v = f2_sub(h, L.eh);
    L.el = f2_add(L.el, f2_add(f2_sub(L.eh, f2_sub(h, v)), f2_sub(er, v)));
    L.eh = h;
}

// The next block of n <= 32 candidates (ring position b) against every lane's atom: |x_j|^2 - 2 x_i x_j <= lim
// (lim = rcut^2 - |x_i|^2 with slack for the rounding); accepted ones are listed per lane. Then hits are
// evaluated while most lanes have two pending, or some lane could run out of room: more than 32 pending (a
// block adds up to 32 to the list's 64), or hits left of the block four before this one (before the next block is
// due, candidates are written up to three blocks short of this one).
__device__ __forceinline__ void rs_block(const RealDev &d, RsWarp &W, RsLane &L, int b, int n, int quorum, unsigned hit0) {
    L.past = (L.past << 8) | ((unsigned)L.cnt & 255u);
    if (L.wp >= hit0 + 64 * 32) {
        L.wrap = L.rp == L.wp ? 0u : L.wp;
        if (L.rp == L.wp) L.rp = hit0;
        L.wp = hit0;
    }
    const unsigned wp0 = L.wp;
    const int f = b & 63;
    const F2 x2 = f2_all(L.xf), y2 = f2_all(L.yf), z2 = f2_all(L.zf);
    auto take = [&](float v, int j) {
        if (v <= L.lim) {
            asm volatile("st.shared.u8 [%0], %1;" ::"r"(L.wp), "r"(j));
            L.wp += 32;
        }
    };
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        if (j < n) {  // uniform
            const float4 X = *(const float4 *)(W.fx + f + j), Y = *(const float4 *)(W.fy + f + j),
                         Z = *(const float4 *)(W.fz + f + j), S = *(const float4 *)(W.f2 + f + j);
            const float2 lo = f2_get(f2_fma(x2, f2(X.x, X.y), f2_fma(y2, f2(Y.x, Y.y), f2_fma(z2, f2(Z.x, Z.y), f2(S.x, S.y)))));
            const float2 hi = f2_get(f2_fma(x2, f2(X.z, X.w), f2_fma(y2, f2(Y.z, Y.w), f2_fma(z2, f2(Z.z, Z.w), f2(S.z, S.w)))));
            take(lo.x, b + j);
            take(lo.y, b + j + 1);
            take(hi.x, b + j + 2);
            take(hi.y, b + j + 3);
        }
    }
    L.cnt += (int)(L.wp - wp0) >> 5;
    while (__popc(__ballot_sync(0xffffffffu, L.cnt - L.done >= 2)) >= quorum ||
           __any_sync(0xffffffffu, L.cnt - L.done > 32 || (signed char)((L.past >> 24) - (unsigned)L.done) > 0))
        rs_evaluate(d, W, L, hit0);
}

// 5: one CTA of NW warps per work item (up to 32 sorted atoms, lane = atom in every warp). The neighbouring
// runs of atoms are laid end to end; each warp takes every NW-th pair of candidates and keeps those within the
// cutoff of the box around the item's atoms in its ring; blocks of 32 are tested against each lane's atom and
// the accepted pairs evaluated lane by lane, so that nearly all lanes evaluate a pair at every step. A load of
// 32 candidates takes 16 pairs from all over the neighbourhood, so that every lane's hits come at about the same
// rate. The warps' sums meet in shared memory in warp order.
//
// 65536 atoms, 9 A cutoff (20 M ordered pairs, 2300 items of 1130 candidates each after the box test): 120 us,
// 84 M warp instructions, issue slots 61 % busy (arithmetic dependencies and shared-memory loads), 18 of 64 warps.
// One thread per atom evaluating every candidate of (2 R + 1)^3 cells as wide as the cutoff, 15 % of them inside
// it, took 794 us. A warp per two atoms with the candidates across the lanes took 170 us, bit masks instead of
// byte lists of hits 138 us, scalar instead of paired FP32 instructions 144 us; 16, 24 or 28 warps per SM instead
// of 20 cost 6, 3 and 4 %.
template <int NW>
__global__ void __launch_bounds__(32 * NW, 20 / NW) k_rs_pairs(RealDev d) {
    extern __shared__ __align__(16) unsigned char smem[];
    RsShared<NW> &Sh = *(RsShared<NW> *)smem;
    pdl_wait();
    if (blockIdx.x >= d.ctl->nitems) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    RsWarp &W = Sh.w[warp];
    const int2 item = d.items[blockIdx.x];
    const bool mine = lane < item.y;
    const int at = item.x + (mine ? lane : 0);
    const int4 me = d.sx[at];
    const int cid0 = d.scell[item.x], cid1 = d.scell[item.x + item.y - 1];
    // centre and half extents of the box around the item's atoms
    const int4 X0 = make_int4(__shfl_sync(0xffffffffu, me.x, 0), __shfl_sync(0xffffffffu, me.y, 0), __shfl_sync(0xffffffffu, me.z, 0), 0);
    RsLane L;
    L.x = wsub(me.x, X0.x);
    L.y = wsub(me.y, X0.y);
    L.z = wsub(me.z, X0.z);
    L.q = __int_as_float(me.w);
    int cx, cy, cz;
    float hx, hy, hz;
    {
        auto box = [](int v, int &c, float &h) {
            const int lo = __reduce_min_sync(0xffffffffu, v), hi = __reduce_max_sync(0xffffffffu, v);
            c = lo + (int)(((unsigned)hi - (unsigned)lo) >> 1);
            h = fmaxf((float)(hi - c), (float)(c - lo)) * 1.000001f;
        };
        box(L.x, cx, hx);
        box(L.y, cy, hy);
        box(L.z, cz, hz);
    }
    L.x -= cx;
    L.y -= cy;
    L.z -= cz;
    cx = wadd(cx, X0.x);
    cy = wadd(cy, X0.y);
    cz = wadd(cz, X0.z);
    L.fx = L.fy = L.fz = L.eh = L.el = f2_all(0.f);
#pragma unroll
    for (int k = 0; k < 6; ++k) L.w[k] = f2_all(0.f);
    const unsigned hit0 = shared_u32(&W.hit[0][lane]);
    L.wp = L.rp = hit0;
    L.wrap = L.past = 0u;
    L.cnt = L.done = 0;
    L.xf = (float)L.x;
    L.yf = (float)L.y;
    L.zf = (float)L.z;
    // the expanded test rounds terms of up to 2 (|h| + rcut)^2 a few times: 2^-19 of that as slack
    const float hh = sqrtf(hx * hx + hy * hy + hz * hz), rc = sqrtf(d.rc2_slack);
    L.lim = mine ? d.rc2_slack + 1.9073486328125e-06f * (hh + rc) * (hh + rc) - fmaf(L.xf, L.xf, fmaf(L.yf, L.yf, L.zf * L.zf))
                 : -3.0e38f;
    const int quorum = item.y - (item.y >> 3);
    if (lane == 0) W.x[0] = make_int4(0, 0, 0, 0);  // what a lane without a hit reads

    // pieces: row offset (o0, o1) and image wz along axis 2, whose cells [za - R2, zb + R2] it contributes
    const int row = cid0 / d.nc[2], za = cid0 - row * d.nc[2], zb = cid1 - row * d.nc[2];
    const int c0 = row / d.nc[1], c1 = row - c0 * d.nc[1];
    const int wz0 = floordiv(za - d.R[2], d.nc[2]), wz1 = floordiv(zb + d.R[2], d.nc[2]);
    const int n1 = 2 * d.R[1] + 1, nz = wz1 - wz0 + 1, np = (2 * d.R[0] + 1) * n1 * nz;
    int head = 0, fresh = 0;  // ring position of the next candidate; candidates not tested yet (the last ones)
    for (int p0 = 0; p0 < np; p0 += 32 * NW) {
        const int p = p0 + tid;
        int cnt = 0;
        RsPiece pc = {0, 0, 0, 0};
        if (p < np) {
            const int pr = p / nz, wz = wz0 + (p - pr * nz);
            const int o0 = pr / n1, u0 = c0 + o0 - d.R[0], u1 = c1 + (pr - o0 * n1) - d.R[1];
            const int w0 = floordiv(u0, d.nc[0]), w1 = floordiv(u1, d.nc[1]);
            const int base = ((u0 - w0 * d.nc[0]) * d.nc[1] + (u1 - w1 * d.nc[1])) * d.nc[2];
            const int lo = max(za - d.R[2] - wz * d.nc[2], 0), hi = min(zb + d.R[2] - wz * d.nc[2], d.nc[2] - 1);
            pc.first = (int)d.start[base + lo];
            cnt = (int)d.start[base + hi + 1] - pc.first;
            pc.sx = wsub(image_offset(d, 0, w0, w1, wz), cx);
            pc.sy = wsub(image_offset(d, 1, w0, w1, wz), cy);
            pc.sz = wsub(image_offset(d, 2, w0, w1, wz), cz);
        }
        int end = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += v;
        }
        if (p0) __syncthreads();  // the previous pieces are done with
        if (lane == 31) Sh.wtot[warp] = end;
        __syncthreads();
        int total = 0;
#pragma unroll
        for (int v = 0; v < NW; ++v) {
            if (v == warp) end += total;
            total += Sh.wtot[v];
        }
        pc.first -= end - cnt;  // candidate c of the pieces is sorted atom first + c
        Sh.piece[tid] = pc;
        Sh.end[tid] = end;
        __syncthreads();
        // candidates in pairs: lanes 2 k, 2 k + 1 take those of [k per, (k + 1) per), every NW-th pair of them. The
        // next load is issued before the current candidates are worked on.
        const int pairs = (total + 1) >> 1, per = (pairs + 15) >> 4;
        int c = 2 * ((lane >> 1) * per + warp) + (lane & 1);
        const int cend = min(2 * min(((lane >> 1) + 1) * per, pairs), total);
        int b = 0, bend;  // the piece: the number of ends <= c
#pragma unroll
        for (int h = 16 * NW; h > 0; h >>= 1)
            if (Sh.end[b + h - 1] <= c) b += h;
        RsPiece q = Sh.piece[b];
        bend = Sh.end[b];
        int4 Jn = make_int4(0, 0, 0, 0);
        if (c < cend) Jn = d.sx[q.first + c];
        for (int i = 0; i < per; i += NW) {
            const bool have = c < cend;
            const int4 J = make_int4(wadd(Jn.x, q.sx), wadd(Jn.y, q.sy), wadd(Jn.z, q.sz), Jn.w);
            c += 2 * NW;
            if (c < cend) {
                if (c >= bend) {  // ends: the last piece ends at total
                    do bend = Sh.end[++b];
                    while (c >= bend);
                    q = Sh.piece[b];
                }
                Jn = d.sx[q.first + c];
            }
            const float jx = (float)J.x, jy = (float)J.y, jz = (float)J.z;
            const float ax = fmaxf(fabsf(jx) - hx, 0.f), ay = fmaxf(fabsf(jy) - hy, 0.f), az = fmaxf(fabsf(jz) - hz, 0.f);
            const bool keep = have && fmaf(ax, ax, fmaf(ay, ay, az * az)) <= d.rc2_slack;
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                int k = head + __popc(m & ((1u << lane) - 1u));
                if (k >= RS_CAND) k -= RS_CAND;
                W.x[k] = J;
                k &= 63;  // RS_CAND is a multiple of 64
                W.fx[k] = -2.f * jx;
                W.fy[k] = -2.f * jy;
                W.fz[k] = -2.f * jz;
                W.f2[k] = fmaf(jx, jx, fmaf(jy, jy, jz * jz));
            }
            head += __popc(m);
            fresh += __popc(m);
            if (head >= RS_CAND) head -= RS_CAND;
            if (fresh >= 32) {
                __syncwarp();
                const int at = head - fresh;  // a multiple of 32
                rs_block(d, W, L, at < 0 ? at + RS_CAND : at, 32, quorum, hit0);
                fresh -= 32;
                __syncwarp();
            }
        }
    }
    __syncwarp();
    {
        const int b = head < fresh ? head - fresh + RS_CAND : head - fresh;
        if (lane >= fresh) {  // the rest of the last block: out of reach
            const int k = (b + lane) & 63;
            W.fx[k] = W.fy[k] = W.fz[k] = 0.f;
            W.f2[k] = 3.0e38f;
        }
        __syncwarp();
        rs_block(d, W, L, b, fresh, quorum, hit0);
    }
    while (__any_sync(0xffffffffu, L.done < L.cnt)) rs_evaluate(d, W, L, hit0);

    // per lane: the warps' sums in warp order; component c of energy / virial by warp c mod NW, over the lanes in
    // a fixed double-float tree
    __syncthreads();
    float(*red)[12][32] = (float(*)[12][32])smem;
    auto both = [](F2 v) {
        const float2 a = f2_get(v);
        return a.x + a.y;
    };
    red[warp][0][lane] = both(L.fx);
    red[warp][1][lane] = both(L.fy);
    red[warp][2][lane] = both(L.fz);
#pragma unroll
    for (int k = 0; k < 6; ++k) red[warp][3 + k][lane] = both(L.w[k]);
    {
        const float2 h = f2_get(L.eh), l = f2_get(L.el);
        DF en = {h.x, l.x}, e2 = {h.y, l.y};
        en = df_add(en, e2);
        red[warp][9][lane] = en.hi;
        red[warp][10][lane] = en.lo;
    }
    __syncthreads();
    for (int k = warp; k < 3; k += NW) {
        float f = 0.f;
#pragma unroll
        for (int v = 0; v < NW; ++v) f += red[v][k][lane];
        if (mine) {
            const float F = f * d.inv_u2;  // exact: a power of two
            float *o = d.forces + 3 * (size_t)d.sidx[at] + k;
            *o = d.accumulate ? *o + F : F;
        }
    }
    for (int k = warp; k < RS_SUMS; k += NW) {
        if (k == 7) {  // the self term, in FP64
            double t = mine ? (double)__int_as_float(me.w) : 0.0;
            t *= t;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            if (lane == 0) d.sums[RS_SUMS * (size_t)blockIdx.x + k] = t;
            continue;
        }
        DF t = {0.f, 0.f};
#pragma unroll
        for (int v = 0; v < NW; ++v) {
            DF a;
            a.hi = k == 0 ? red[v][9][lane] : red[v][2 + k][lane];
            a.lo = k == 0 ? red[v][10][lane] : 0.f;
            t = df_add(t, a);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            DF a;
            a.hi = __shfl_down_sync(0xffffffffu, t.hi, o);
            a.lo = __shfl_down_sync(0xffffffffu, t.lo, o);
            t = df_add(t, a);
        }
        if (lane == 0) d.sums[RS_SUMS * (size_t)blockIdx.x + k] = (double)t.hi + (double)t.lo;
    }
}

// FP64 sums of rows of RS_SUMS values, 256 threads: thread t adds value t mod 8 of the rows [b, e) from b + t / 8 in
// steps of 32, then the 32 partial sums meet in a fixed tree; out[k] (shared or global) by threads k < 8.
__device__ __forceinline__ void sum_rows(const double *rows, int b, int e, double *out) {
    __shared__ double wsum[8][RS_SUMS];
    const int tid = threadIdx.x, k = tid & 7;
    double v = 0.0;
    for (int a = b + (tid >> 3); a < e; a += 32) v += __ldcg(rows + RS_SUMS * (size_t)a + k);
    v += __shfl_down_sync(0xffffffffu, v, 16);
    v += __shfl_down_sync(0xffffffffu, v, 8);
    if ((tid & 31) < 8) wsum[tid >> 5][k] = v;
    __syncthreads();
    if (tid < 8) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += wsum[w][tid];
        out[tid] = s;
    }
    __syncthreads();
}

// 6: the work items' sums, in contiguous chunks per block; the block that finishes last adds the blocks' sums in
// order and stores energies, self term and virial in the control block, in d.ev and in d.file. Eight threads
// share a row, one value each, since FP64 additions are slow (a thread per row with all values took 12 us at 2300
// items).
__global__ void __launch_bounds__(256) k_rs_reduce(RealDev d) {
    __shared__ bool last;
    __shared__ double tot[RS_SUMS];
    pdl_wait();
    const int tid = threadIdx.x, nitems = d.n > 0 ? (int)d.ctl->nitems : 0;
    const int chunk = (nitems + gridDim.x - 1) / gridDim.x, b = blockIdx.x * chunk;
    sum_rows(d.sums, b, min(nitems, b + chunk), d.partials + RS_SUMS * blockIdx.x);
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&d.ctl->arrived, 1u) == gridDim.x - 1u;
    __syncthreads();
    if (!last) return;
    __threadfence();
    sum_rows(d.partials, 0, (int)gridDim.x, tot);
    if (tid < 8) {
        // E_real, E_self, virial
        const double sqrt_pi = 1.7724538509055160273;
        const double r = tid == 0 ? 0.5 * tot[0] * d.inv_u
                                  : (tid == 1 ? -d.beta_d / sqrt_pi * tot[7] : 0.5 * tot[tid - 1] * d.inv_u);
        d.ctl->res[tid] = r;
        if (d.ev) d.ev[tid] = r;
        if (d.host) {
            d.host->res[tid] = r;
            if (tid == 0) d.host->status = __ldcg(&d.ctl->status);
        }
        if (d.file_step) {
            const unsigned step = *d.file_step;
            if (d.file && step < (unsigned)d.file_rows) d.file[(size_t)step * d.file_stride + tid] = r;
            __syncwarp(0xffu);
            if (tid == 0) *d.file_step = step + 1u;
        }
    }
    if (tid == 0) d.ctl->arrived = 0u;
}

}  // namespace pme

using namespace pme;

struct pme_real {
    int dev = 0;
    cudaStream_t stream = nullptr;
    double box[9] = {0}, recip[9] = {0}, vol = 0.0, beta = 0.0, rcut = 0.0;
    RealDev d;
    RealGrid fine, coarse;     // the cells for many and for few atoms (real_grid)
    void *cell_mem = nullptr;  // counts, starts, partials, control block (per box)
    size_t cell_bytes = 0;
    void *atom_mem = nullptr;  // per-atom scratch (grows with n)
    size_t atom_bytes = 0;
    int64_t n_cap = 0;
    RealCtl *h_ctl = nullptr, *h_ctl_dev = nullptr;  // page-locked results of the synchronous call
    unsigned long long gen = 0;  // bumped whenever the kernels' arguments change (cell, scratch)
};

static size_t al256r(size_t x) { return (x + 255) & ~(size_t)255; }

// Cells narrower than the cutoff by the factor sub (sub of them along axes the cutoff spans), in rows along axis 2
// that are cut into slabs of about `slab` cells, which bounds a work item's extent. The unit u is the smallest power of
// two with 2^31 u above every coordinate difference a work item forms: its own extent, R cells and one more.
static double real_cells(const double box[9], const double recip[9], double rcut, int sub, int slab, RealGrid &d) {
    double ncells = 1.0;
    for (int al = 0; al < 3; ++al) {
        const double astar = sqrt(recip[3 * al] * recip[3 * al] + recip[3 * al + 1] * recip[3 * al + 1] +
                                  recip[3 * al + 2] * recip[3 * al + 2]);
        const double wfrac = rcut * astar * (1.0 + 1e-6);
        d.nc[al] = wfrac < 1.0 ? (int)std::min(floor(sub / wfrac), 1e9) : sub;
        d.R[al] = std::max(1, (int)ceil(wfrac * d.nc[al] - 1e-12));
        ncells *= d.nc[al];
    }
    d.ncells = ncells <= RS_MAX_CELLS ? (int)ncells : 0;
    d.nslab = std::max(1, (d.nc[2] + slab / 2) / slab);
    d.slab = (d.nc[2] + d.nslab - 1) / d.nslab;
    d.nslab = (d.nc[2] + d.slab - 1) / d.slab;
    d.nrowslabs = d.ncells ? d.nc[0] * d.nc[1] * d.nslab : 0;
    double most = 0.0;
    for (int k = 0; k < 3; ++k) {
        double b = 0.0;
        for (int al = 0; al < 3; ++al)
            b += fabs(box[3 * al + k]) * ((al == 2 ? d.slab : 1) + d.R[al] + 1) / d.nc[al];
        most = std::max(most, b);
    }
    int e;
    frexp(most * 1.001, &e);  // below 2^e
    d.inv_u = ldexp(1.0, 31 - e);
    return ncells;
}

// The grid's constants that follow from its unit.
static void real_units(const double box[9], const double recip[9], double beta, double rcut, RealGrid &d) {
    for (int al = 0; al < 3; ++al)
        for (int j = 0; j < 3; ++j) {
            d.rec[3 * al + j] = (float)recip[3 * al + j];
            const double v = box[3 * al + j] * d.inv_u, i = rint(v);
            d.afix[3 * al + j] = (int)(unsigned)(unsigned long long)(long long)i;
            d.afrac[3 * al + j] = (float)(v - i);
        }
    const double u = 1.0 / d.inv_u, rcu = rcut * d.inv_u;
    d.inv_u2 = (float)(d.inv_u * d.inv_u);
    d.rc2 = (float)(rcu * rcu);
    d.rc2_slack = (float)(rcu * rcu * (1.0 + 2e-5));
    d.beta04_u = (float)(0.4 * beta * u);
    d.ex_k = (float)(beta * beta * u * u * 1.4426950408889634074);
    d.c2_u = (float)(2.0 * beta * u / 1.7724538509055160273);
}

// The cells for n atoms: about half a cutoff wide, so that the neighbouring cells -R..R hug the cutoff sphere (3.7
// instead of 6.4 candidates per pair inside the cutoff), where there are no more of them than atoms; at least a cutoff
// wide otherwise, or where the box has more than RS_MAX_CELLS of the others. With fewer atoms than cells, the scan of
// the cells and work items of an atom or two are what counts: us with fine / coarse cells, and of one thread per atom
// over coarse cells, for 65536 atoms, 9 A cutoff, 0.9 atoms in a fine cell 109 / 58, 174; 0.09 549 / 120, 190; 5 A, 0.2
// 366 / 92, 150; 2048 atoms, 9 A, 0.09 48 / 24, 65. The line would lie at about 4 for uniform systems (2.7 atoms 96 / 74,
// 6.5 atoms at 12 A 117 / 122), but a droplet's neighbourhoods are full whatever its mean (8 times the mean, 2.7 atoms
// at 12 A: 219 / 251). The atom count alone decides, so a system's sums depend on nothing else.
static const RealGrid &real_grid(const pme_real *rs, int64_t n) {
    return rs->fine.ncells && n >= rs->fine.ncells ? rs->fine : rs->coarse;
}
// The kernels' arguments for n atoms, but for the caller's arrays.
static RealDev real_args(const pme_real *rs, int64_t n) {
    RealDev d = rs->d;
    (RealGrid &)d = real_grid(rs, n);
    d.n = (int)n;
    return d;
}

// Checks the cutoff against the box and sets the cell grids; PME_EUNSUPPORTED when rcut needs more than RS_MAX_R cells
// per axis or the grid of cells at least a cutoff wide has more than RS_MAX_CELLS.
static pme_status real_geometry(pme_real *rs, const double box[9]) {
    double recip[9], vol;
    if (!cell_reciprocal(box, recip, &vol)) return fail(PME_EINVAL, "box is singular");
    RealGrid fine, coarse;
    // slabs of ten cutoffs, so that both grids have about the same unit
    const double nfine = real_cells(box, recip, rs->rcut, 2, 20, fine);
    const double ncells = real_cells(box, recip, rs->rcut, 1, nfine <= RS_MAX_CELLS ? 10 : 20, coarse);
    for (int al = 0; al < 3; ++al)
        if (coarse.R[al] > RS_MAX_R)
            return fail(PME_EUNSUPPORTED, "rcut %.3g A spans %d cell widths along axis %d (at most %d)", rs->rcut, coarse.R[al],
                        al, RS_MAX_R);
    if (ncells > RS_MAX_CELLS) return fail(PME_EUNSUPPORTED, "%.0f cells (at most %d): rcut too small for this box", ncells, RS_MAX_CELLS);
    memcpy(rs->box, box, sizeof(rs->box));
    memcpy(rs->recip, recip, sizeof(recip));
    rs->vol = vol;
    real_units(box, recip, rs->beta, rs->rcut, fine);
    real_units(box, recip, rs->beta, rs->rcut, coarse);
    rs->fine = fine;
    rs->coarse = coarse;
    return PME_OK;
}

static pme_status real_alloc_cells(pme_real *rs) {
    const size_t nc = (size_t)std::max(rs->fine.ncells, rs->coarse.ncells);
    size_t off = 0;
    const size_t o_cnt = off;  off = al256r(off + nc * 4);
    const size_t o_st = off;   off = al256r(off + (nc + 1) * 4);
    const size_t o_par = off;  off = al256r(off + RS_RED_BLOCKS * RS_SUMS * sizeof(double));
    const size_t o_ctl = off;  off = al256r(off + sizeof(RealCtl));
    if (off > rs->cell_bytes) {
        if (rs->cell_mem) cudaFree(rs->cell_mem);
        rs->cell_mem = nullptr;
        rs->cell_bytes = 0;
        cudaError_t e = lib_malloc(&rs->cell_mem, off);
        if (e != cudaSuccess) {
            rs->cell_mem = nullptr;
            return fail(PME_ENOMEM, "cudaMalloc(%zu bytes): %s", off, cudaGetErrorString(e));
        }
        rs->cell_bytes = off;
    }
    cudaError_t e = cudaMemsetAsync(rs->cell_mem, 0, rs->cell_bytes, rs->stream);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync(cells)");
    char *b = (char *)rs->cell_mem;
    RealDev &d = rs->d;
    d.count = (unsigned *)(b + o_cnt);
    d.start = (unsigned *)(b + o_st);
    d.partials = (double *)(b + o_par);
    d.ctl = (RealCtl *)(b + o_ctl);
    return PME_OK;
}

static pme_status real_reserve(pme_real *rs, int64_t n) {
    if (n <= rs->n_cap && rs->atom_mem) return PME_OK;
    const size_t m = (size_t)(n > 0 ? n : 1);
    size_t off = 0;
    const size_t o_cell = off; off = al256r(off + m * 8);
    const size_t o_xq = off;   off = al256r(off + m * 16);
    const size_t o_aidx = off; off = al256r(off + m * 4);
    const size_t o_sx = off;   off = al256r(off + m * 16);
    const size_t o_sidx = off; off = al256r(off + m * 4);
    const size_t o_sc = off;   off = al256r(off + m * 4);
    const size_t o_it = off;   off = al256r(off + m * 8);
    const size_t o_sum = off;  off = al256r(off + m * RS_SUMS * 8);
    const size_t o_own = off;  off = al256r(off + m * 12);
    cudaError_t e = cudaStreamSynchronize(rs->stream);
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    if (rs->atom_mem) cudaFree(rs->atom_mem);
    rs->atom_mem = nullptr;
    rs->atom_bytes = 0;
    rs->n_cap = 0;
    if ((e = lib_malloc(&rs->atom_mem, off)) != cudaSuccess) {
        rs->atom_mem = nullptr;
        return fail(PME_ENOMEM, "cudaMalloc(%zu bytes): %s", off, cudaGetErrorString(e));
    }
    char *b = (char *)rs->atom_mem;
    RealDev &d = rs->d;
    d.cell = (int2 *)(b + o_cell);
    d.xq = (int4 *)(b + o_xq);
    d.aidx = (int *)(b + o_aidx);
    d.sx = (int4 *)(b + o_sx);
    d.sidx = (int *)(b + o_sidx);
    d.scell = (int *)(b + o_sc);
    d.items = (int2 *)(b + o_it);
    d.sums = (double *)(b + o_sum);
    d.fown = (float *)(b + o_own);
    rs->atom_bytes = off;
    rs->n_cap = (int64_t)m;
    ++rs->gen;
    return PME_OK;
}

// Chained by programmatic dependent launch: every kernel waits for its predecessor before it touches data.
static void rs_launch(void (*kernel)(RealDev), unsigned grid, unsigned block, size_t smem, cudaStream_t s, const RealDev &d) {
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
    cudaLaunchKernelEx(&cfg, kernel, d);
}

// Warps per work item. An item needs about 28 atoms' worth of a CTA, so small systems have few CTAs and gain
// from more warps in each; large ones fill the GPU with either and evaluate with fewer idle lanes when a warp
// sees more of the candidates. Measured with 4 / 8 / 16 warps (us): real space of 2048 atoms 66 / 58 / 54, of 3500
// - / 50 / 45, of 18000 76 / 82 / -; 32 MD steps of 8190 atoms 2338 / 2019 / 2180, of 12000 1866 / 1692 / -, of 18000
// 1952 / 2102 / -; full Ewald of 65536 atoms 169 / 193 / 235. (Six warps, three CTAs per SM, for 300 to 456 items: 32
// steps of 8190 atoms 1424 against 1199 with eight.) All at liquid density: what counts is the number of items, and a
// gas has more of them for its atoms (2048 atoms at 0.0001 / A^3, 9 A: 62 with 16 warps, 34 with two; 84 with one thread
// per atom). A system's sums depend on the number of warps, hence on the atom count alone.
static int rs_pair_warps(const RealDev &d) { return d.n <= 4096 ? 16 : (d.n <= 15000 ? 8 : 4); }

static void launch_pairs(const RealDev &d0, cudaStream_t s) {
    RealDev d = d0;
    const unsigned g = (unsigned)((d.n + 255) / 256);
    d.max_items = d.n / 32 + std::min(d.n, d.nrowslabs);
    if (d.n < 1) return;
    rs_launch(k_rs_bin, (unsigned)((d.n + RS_BIN_THREADS - 1) / RS_BIN_THREADS), RS_BIN_THREADS, 0, s, d);
    rs_launch(k_rs_scan, 1, RS_SCAN_THREADS, 0, s, d);
    rs_launch(k_rs_scatter, g, 256, 0, s, d);
    rs_launch(k_rs_rank, g, 256, 0, s, d);
    const int warps = rs_pair_warps(d);
    if (warps == 4) rs_launch(k_rs_pairs<4>, (unsigned)d.max_items, 128, sizeof(RsShared<4>), s, d);
    else if (warps == 8) rs_launch(k_rs_pairs<8>, (unsigned)d.max_items, 256, sizeof(RsShared<8>), s, d);
    else rs_launch(k_rs_pairs<16>, (unsigned)d.max_items, 512, sizeof(RsShared<16>), s, d);
}

static void launch_reduce(const RealDev &d, cudaStream_t s) { rs_launch(k_rs_reduce, RS_RED_BLOCKS, 256, 0, s, d); }

extern "C" {

pme_status pme_real_create(const double box[9], double beta, double rcut, void *cuda_stream, pme_real **out) {
    if (!out) return fail(PME_EINVAL, "out is NULL");
    *out = nullptr;
    if (!box) return fail(PME_EINVAL, "box is NULL");
    if (!(beta > 0.0) || !isfinite(beta) || !(rcut > 0.0) || !isfinite(rcut))
        return fail(PME_EINVAL, "beta and rcut must be positive and finite");
    for (int i = 0; i < 9; ++i)
        if (!isfinite(box[i])) return fail(PME_EINVAL, "box has a non-finite entry");
    pme_real *rs = lib_new<pme_real>();
    if (!rs) return fail(PME_ENOMEM, "host allocation failed");
    cudaError_t e = cudaGetDevice(&rs->dev);
    if (e != cudaSuccess) {
        delete rs;
        return cuda_fail(e, "cudaGetDevice");
    }
    rs->stream = (cudaStream_t)cuda_stream;
    rs->beta = beta;
    rs->rcut = rcut;
    memset(&rs->d, 0, sizeof(rs->d));
    rs->d.beta_d = beta;
    if ((e = cudaFuncSetAttribute((const void *)k_rs_pairs<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RsShared<4>))) != cudaSuccess ||
        (e = cudaFuncSetAttribute((const void *)k_rs_pairs<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RsShared<8>))) != cudaSuccess ||
        (e = cudaFuncSetAttribute((const void *)k_rs_pairs<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RsShared<16>))) != cudaSuccess) {
        delete rs;
        return cuda_fail(e, "configure the pair kernels");
    }
    pme_status st;
    if ((st = real_geometry(rs, box)) != PME_OK || (st = real_alloc_cells(rs)) != PME_OK ||
        (st = real_reserve(rs, 1)) != PME_OK) {
        pme_real_destroy(rs);
        return st;
    }
    if ((e = lib_malloc_host((void **)&rs->h_ctl, sizeof(RealCtl))) != cudaSuccess) {
        rs->h_ctl = nullptr;
        pme_real_destroy(rs);
        return cuda_fail(e, "cudaMallocHost");
    }
    memset(rs->h_ctl, 0, sizeof(RealCtl));
    if ((e = cudaHostGetDevicePointer((void **)&rs->h_ctl_dev, rs->h_ctl, 0)) != cudaSuccess) {
        pme_real_destroy(rs);
        return cuda_fail(e, "cudaHostGetDevicePointer");
    }
    if ((e = cudaStreamSynchronize(rs->stream)) != cudaSuccess) {
        pme_real_destroy(rs);
        return cuda_fail(e, "cudaStreamSynchronize");
    }
    *out = rs;
    return PME_OK;
}

pme_status pme_real_set_box(pme_real *rs, const double box[9]) {
    if (!rs || !box) return fail(PME_EINVAL, "real-space context and box must be non-NULL");
    for (int i = 0; i < 9; ++i)
        if (!isfinite(box[i])) return fail(PME_EINVAL, "box has a non-finite entry");
    DeviceGuard g(rs->dev);
    cudaError_t e = cudaStreamSynchronize(rs->stream);
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    pme_status st = real_geometry(rs, box);
    if (st != PME_OK) return st;
    ++rs->gen;
    if ((st = real_alloc_cells(rs)) != PME_OK) return st;
    if ((e = cudaStreamSynchronize(rs->stream)) != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    return PME_OK;
}

pme_status pme_real_reserve(pme_real *rs, int64_t n) {
    if (!rs) return fail(PME_EINVAL, "real-space context is NULL");
    if (n < 0 || n > (int64_t)0x3fffffff) return fail(PME_EINVAL, "n out of range");
    DeviceGuard g(rs->dev);
    return real_reserve(rs, n);
}

pme_status pme_real_enqueue(pme_real *rs, const float *pos, const float *q, int64_t n, float *forces, int accumulate,
                            double *ev_dev) {
    if (!rs) return fail(PME_EINVAL, "real-space context is NULL");
    return real_enqueue_on(rs, rs->stream, pos, q, n, forces, accumulate, ev_dev);
}

}  // extern "C"

// The same on a given stream (the multi-step loop runs everything on its plan's stream).
pme_status pme::real_enqueue_on(pme_real *rs, cudaStream_t stream, const float *pos, const float *q, int64_t n,
                                float *forces, int accumulate, double *ev_dev) {
    if (n < 0 || n > (int64_t)0x3fffffff) return fail(PME_EINVAL, "n = %lld out of range [0, 2^30)", (long long)n);
    if (n > 0 && (!pos || !q || !forces)) return fail(PME_EINVAL, "pos, q and forces must be non-NULL when n > 0");
    DeviceGuard g(rs->dev);
    pme_status st = real_reserve(rs, n);
    if (st != PME_OK) return st;
    RealDev d = real_args(rs, n);
    d.pos = pos;
    d.q = q;
    d.forces = forces;
    d.accumulate = accumulate ? 1 : 0;
    d.ev = ev_dev;
    launch_pairs(d, stream);
    launch_reduce(d, stream);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "real-space kernel launch");
    return PME_OK;
}

// The evaluation into the context's own force array, in two parts: forces (the array is returned; n has been
// reserved), then energies, filed as one row of a table per call.
const float *pme::real_enqueue_own(pme_real *rs, cudaStream_t stream, const float *pos, const float *q, int64_t n) {
    RealDev d = real_args(rs, n);
    d.pos = pos;
    d.q = q;
    d.forces = d.fown;
    launch_pairs(d, stream);
    return d.fown;
}
void pme::real_enqueue_file(pme_real *rs, cudaStream_t stream, int64_t n, unsigned *step, double *file, int stride, int rows) {
    RealDev d = real_args(rs, n);
    d.file_step = step;
    d.file = file;
    d.file_stride = stride;
    d.file_rows = rows;
    launch_reduce(d, stream);
}

pme_status pme::real_reserve_n(pme_real *rs, int64_t n) {
    DeviceGuard g(rs->dev);
    return real_reserve(rs, n);
}

int pme::real_device(const pme_real *rs) { return rs->dev; }
unsigned long long pme::real_gen(const pme_real *rs) { return rs->gen; }

extern "C" {

pme_status pme_real_compute(pme_real *rs, const float *pos, const float *q, int64_t n, float *forces,
                            double *e_real, double *e_self, double *virial) {
    if (!rs) return fail(PME_EINVAL, "real-space context is NULL");
    // the reduction stores the results and the status word in page-locked memory itself (a copy-engine transfer
    // of the block after it took 7 us more: 2048 atoms, 52 -> 45 us)
    rs->d.host = rs->h_ctl_dev;
    pme_status st = real_enqueue_on(rs, rs->stream, pos, q, n, forces, 0, nullptr);
    rs->d.host = nullptr;
    if (st != PME_OK) return st;
    DeviceGuard g(rs->dev);
    cudaError_t e;
    if ((e = cudaStreamSynchronize(rs->stream)) != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    const unsigned bits = rs->h_ctl->status;
    if (bits) {
        cudaMemsetAsync(&rs->d.ctl->status, 0, sizeof(unsigned), rs->stream);
        cudaStreamSynchronize(rs->stream);
        return status_from_bits(bits);
    }
    if (e_real) *e_real = rs->h_ctl->res[0];
    if (e_self) *e_self = rs->h_ctl->res[1];
    if (virial)
        for (int k = 0; k < 6; ++k) virial[k] = rs->h_ctl->res[2 + k];
    return PME_OK;
}

void pme_real_destroy(pme_real *rs) {
    if (!rs) return;
    DeviceGuard g(rs->dev);
    cudaStreamSynchronize(rs->stream);
    if (rs->cell_mem) cudaFree(rs->cell_mem);
    if (rs->atom_mem) cudaFree(rs->atom_mem);
    if (rs->h_ctl) cudaFreeHost(rs->h_ctl);
    delete rs;
}

}  // extern "C"
