// Batched complex FFTs in shared memory (Stockham auto-sort, mixed radix 2/3/4/5/8).
//
// The paper builds its 3D FFT from pipelined radix-2 1D FFT units (Sec. III-B, Sec. IV-A). On a GPU the
// 1D transforms of a slab or pencil instead live in shared memory: each stage reads R points at stride
// N/R, applies the twiddles W_{Ns R}^{r k}, does a radix-R DFT in registers, and writes the R outputs at
// stride Ns, ping-ponging between two buffers. Input and output are in natural order, so no bit-reversal
// pass and no permuted tables are needed. Lengths are any product of 2, 3, 5 up to 128.
//
// Sign convention: forward = exp(-2 pi i jk/N), inverse = exp(+2 pi i jk/N), both unnormalised.
#pragma once

#include "common.cuh"

namespace pme {

PME_DEV float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
PME_DEV float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
PME_DEV float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
PME_DEV float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
PME_DEV float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// multiply by -i (forward) or +i (inverse)
template <bool INV>
PME_DEV float2 cmul_mi(float2 a) {
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

template <int R, bool INV>
PME_DEV void dft_small(float2 *v);

template <>
PME_DEV void dft_small<2, false>(float2 *v) {
    float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
}
template <>
PME_DEV void dft_small<2, true>(float2 *v) {
    dft_small<2, false>(v);
}

template <bool INV>
PME_DEV void dft4(float2 &a0, float2 &a1, float2 &a2, float2 &a3) {
    float2 s02 = cadd(a0, a2), d02 = csub(a0, a2);
    float2 s13 = cadd(a1, a3), d13 = cmul_mi<INV>(csub(a1, a3));
    a0 = cadd(s02, s13);
    a2 = csub(s02, s13);
    a1 = cadd(d02, d13);
    a3 = csub(d02, d13);
}

template <>
PME_DEV void dft_small<4, false>(float2 *v) {
    dft4<false>(v[0], v[1], v[2], v[3]);
}
template <>
PME_DEV void dft_small<4, true>(float2 *v) {
    dft4<true>(v[0], v[1], v[2], v[3]);
}

template <bool INV>
PME_DEV void dft8(float2 *v) {
    // even / odd split into two length-4 DFTs, then the W8^k combine
    float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<INV>(e0, e1, e2, e3);
    dft4<INV>(o0, o1, o2, o3);
    const float h = 0.70710678118654752440f;
    // W8^1 = (h, -h) forward, (h, h) inverse; W8^2 = -i / +i; W8^3 = (-h, -h) forward, (-h, h) inverse
    float2 t1 = INV ? make_float2(h * (o1.x - o1.y), h * (o1.x + o1.y)) : make_float2(h * (o1.x + o1.y), h * (o1.y - o1.x));
    float2 t2 = cmul_mi<INV>(o2);
    float2 t3 = INV ? make_float2(-h * (o3.x + o3.y), h * (o3.x - o3.y)) : make_float2(h * (o3.y - o3.x), -h * (o3.x + o3.y));
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, t1);
    v[5] = csub(e1, t1);
    v[2] = cadd(e2, t2);
    v[6] = csub(e2, t2);
    v[3] = cadd(e3, t3);
    v[7] = csub(e3, t3);
}
template <>
PME_DEV void dft_small<8, false>(float2 *v) {
    dft8<false>(v);
}
template <>
PME_DEV void dft_small<8, true>(float2 *v) {
    dft8<true>(v);
}

template <bool INV>
PME_DEV void dft3(float2 *v) {
    const float c = -0.5f, s = 0.86602540378443864676f;  // cos(2 pi/3), sin(2 pi/3)
    float2 a0 = v[0], t1 = cadd(v[1], v[2]), t2 = csub(v[1], v[2]);
    float2 m = make_float2(a0.x + c * t1.x, a0.y + c * t1.y);
    float2 r = cmul_mi<INV>(cscale(t2, s));  // -i s t2 (forward)
    v[0] = cadd(a0, t1);
    v[1] = cadd(m, r);
    v[2] = csub(m, r);
}
template <>
PME_DEV void dft_small<3, false>(float2 *v) {
    dft3<false>(v);
}
template <>
PME_DEV void dft_small<3, true>(float2 *v) {
    dft3<true>(v);
}

template <bool INV>
PME_DEV void dft5(float2 *v) {
    const float c1 = 0.30901699437494742410f, s1 = 0.95105651629515357212f;   // cos, sin(2 pi/5)
    const float c2 = -0.80901699437494742410f, s2 = 0.58778525229247312917f;  // cos, sin(4 pi/5)
    float2 a0 = v[0];
    float2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    float2 t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
    float2 m1 = make_float2(a0.x + c1 * t1.x + c2 * t2.x, a0.y + c1 * t1.y + c2 * t2.y);
    float2 m2 = make_float2(a0.x + c2 * t1.x + c1 * t2.x, a0.y + c2 * t1.y + c1 * t2.y);
    float2 r1 = cmul_mi<INV>(make_float2(s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y));
    float2 r2 = cmul_mi<INV>(make_float2(s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y));
    v[0] = cadd(a0, cadd(t1, t2));
    v[1] = cadd(m1, r1);
    v[4] = csub(m1, r1);
    v[2] = cadd(m2, r2);
    v[3] = csub(m2, r2);
}
template <>
PME_DEV void dft_small<5, false>(float2 *v) {
    dft5<false>(v);
}
template <>
PME_DEV void dft_small<5, true>(float2 *v) {
    dft5<true>(v);
}

// Length 6 as 3 x 2 (Cooley-Tukey): DFT3 of the even and of the odd points, twiddles W6^k, then DFT2.
template <bool INV>
PME_DEV void dft6(float2 *v) {
    float2 a[3] = {v[0], v[2], v[4]}, b[3] = {v[1], v[3], v[5]};
    dft3<INV>(a);
    dft3<INV>(b);
    const float s = 0.86602540378443864676f;  // sin(pi / 3)
    // W6^1 = (1/2, -s) forward, (1/2, s) inverse; W6^2 = (-1/2, -s) forward, (-1/2, s) inverse
    const float sg = INV ? s : -s;
    b[1] = cmul(b[1], make_float2(0.5f, sg));
    b[2] = cmul(b[2], make_float2(-0.5f, sg));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[k] = cadd(a[k], b[k]);
        v[k + 3] = csub(a[k], b[k]);
    }
}
template <>
PME_DEV void dft_small<6, false>(float2 *v) {
    dft6<false>(v);
}
template <>
PME_DEV void dft_small<6, true>(float2 *v) {
    dft6<true>(v);
}

// Length 9 as 3 x 3: DFT3 of the points 0 3 6, 1 4 7, 2 5 8, twiddles W9^{jk}, then DFT3 over j.
template <bool INV>
PME_DEV void dft9(float2 *v) {
    // cos, sin of 2 pi k / 9, k = 1, 2, 4
    const float c1 = 0.76604444311897803520f, s1 = 0.64278760968653932632f;
    const float c2 = 0.17364817766693034885f, s2 = 0.98480775301220805937f;
    const float c4 = -0.93969262078590838405f, s4 = 0.34202014332566873304f;
    float2 a[3][3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        a[j][0] = v[j];
        a[j][1] = v[j + 3];
        a[j][2] = v[j + 6];
        dft3<INV>(a[j]);
    }
    const float sg = INV ? 1.0f : -1.0f;
    a[1][1] = cmul(a[1][1], make_float2(c1, sg * s1));
    a[1][2] = cmul(a[1][2], make_float2(c2, sg * s2));
    a[2][1] = cmul(a[2][1], make_float2(c2, sg * s2));
    a[2][2] = cmul(a[2][2], make_float2(c4, sg * s4));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float2 b[3] = {a[0][k], a[1][k], a[2][k]};
        dft3<INV>(b);
        v[k] = b[0];
        v[k + 3] = b[1];
        v[k + 6] = b[2];
    }
}
template <>
PME_DEV void dft_small<9, false>(float2 *v) {
    dft9<false>(v);
}
template <>
PME_DEV void dft_small<9, true>(float2 *v) {
    dft9<true>(v);
}

// Length 10 as 5 x 2: DFT5 of the even and of the odd points, twiddles W10^k, then DFT2.
template <bool INV>
PME_DEV void dft10(float2 *v) {
    float2 a[5] = {v[0], v[2], v[4], v[6], v[8]}, b[5] = {v[1], v[3], v[5], v[7], v[9]};
    dft5<INV>(a);
    dft5<INV>(b);
    const float sg = INV ? 1.0f : -1.0f;
    // cos, sin of pi k / 5
    b[1] = cmul(b[1], make_float2(0.80901699437494742410f, sg * 0.58778525229247312917f));
    b[2] = cmul(b[2], make_float2(0.30901699437494742410f, sg * 0.95105651629515357212f));
    b[3] = cmul(b[3], make_float2(-0.30901699437494742410f, sg * 0.95105651629515357212f));
    b[4] = cmul(b[4], make_float2(-0.80901699437494742410f, sg * 0.58778525229247312917f));
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        v[k] = cadd(a[k], b[k]);
        v[k + 5] = csub(a[k], b[k]);
    }
}
template <>
PME_DEV void dft_small<10, false>(float2 *v) {
    dft10<false>(v);
}
template <>
PME_DEV void dft_small<10, true>(float2 *v) {
    dft10<true>(v);
}

#if defined(PME_HOST_EMULATION)
// Radix chosen for the remaining length rem = N / Ns: 8, then 4, 2, 3, 5.
PME_DEV int fft_radix(int rem) {
    if (rem % 8 == 0) return 8;
    if (rem % 4 == 0) return 4;
    if (rem % 2 == 0) return 2;
    if (rem % 3 == 0) return 3;
    return 5;
}

// One Stockham stage of radix R over ntr transforms of length N (element e of transform t at
// t*bs + e*es in both buffers). tw[k] = exp(-2 pi i k / N), k < N.
template <int R, bool INV>
PME_DEV void fft_stage(const float2 *src, float2 *dst, int N, int Ns, int ntr, int es, int bs, const float2 *tw) {
    const int nb = N / R;           // butterflies per transform
    const int total = ntr * nb;
    const int tstep = nb / Ns;      // = N / (Ns R): twiddle index step
    const float inv_nb = 1.0f / (float)nb, inv_ntr = 1.0f / (float)ntr, inv_ns = 1.0f / (float)Ns;
    for (int idx = PME_TID; idx < total; idx += PME_NTH) {
        int t, j;
        if (es == 1) {  // rows contiguous: consecutive threads walk one transform
            t = fdiv(idx, inv_nb);
            j = idx - t * nb;
        } else {        // columns: consecutive threads walk consecutive transforms
            j = fdiv(idx, inv_ntr);
            t = idx - j * ntr;
        }
        const float2 *s = src + t * bs;
        float2 *o = dst + t * bs;
        const int jq = fdiv(j, inv_ns);
        const int k = j - jq * Ns;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = s[(j + r * nb) * es];
        if (Ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                float2 w = tw[r * k * tstep];
                if (INV) w.y = -w.y;
                v[r] = cmul(v[r], w);
            }
        }
        dft_small<R, INV>(v);
        const int od = jq * Ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) o[(od + r * Ns) * es] = v[r];
    }
}

// Full transforms; returns the buffer (a or b) that holds the result. Ends with a barrier.
template <bool INV>
PME_DEV float2 *fft_batch(float2 *a, float2 *b, int N, int ntr, int es, int bs, const float2 *tw) {
    int Ns = 1;
    while (Ns < N) {
        const int R = fft_radix(N / Ns);
        switch (R) {
            case 8: fft_stage<8, INV>(a, b, N, Ns, ntr, es, bs, tw); break;
            case 4: fft_stage<4, INV>(a, b, N, Ns, ntr, es, bs, tw); break;
            case 2: fft_stage<2, INV>(a, b, N, Ns, ntr, es, bs, tw); break;
            case 3: fft_stage<3, INV>(a, b, N, Ns, ntr, es, bs, tw); break;
            default: fft_stage<5, INV>(a, b, N, Ns, ntr, es, bs, tw); break;
        }
        PME_SYNC();
        float2 *t = a;
        a = b;
        b = t;
        Ns *= R;
    }
    return a;
}
#endif

// The lane transforms need a warp; PME_EMULATE_WARP says that the including file supplies one on the CPU.
#if !defined(PME_HOST_EMULATION) || defined(PME_EMULATE_WARP)
// ---------------------------------------------------------------------------------------------------------
// Lane-distributed transforms in registers, for lengths N = L * E, L lanes of E points (the lane plans,
// PME_LANE_CASES). The L lanes of one transform sit in one warp at lane ids t + T j (T = floor(32 / L)
// transforms per warp, j = 0 .. L - 1; the 32 - T L lanes left over work on a copy of some transform), so a
// transform's lanes exchange values with shuffles and no CTA barrier. Lane j holds the E points x[j + L n],
// n < E, and the four-step factorisation N = E x L runs as:
//   1. an E-point DFT in each lane over n:          y_j[k] = sum_n x[j + L n] W_E^{n k}
//   2. twiddles:                                    y_j[k] *= W_N^{j k}
//   3. an L-point DFT across lanes over j, by decimation in frequency: a round on groups of M lanes (M = L, then
//      M = h, ...) takes the radix r = 5, 3 or 2, the first that divides M, and with h = M / r turns lane
//      j = p h + s of a group (p < r, s < h) into W_M^{p s} sum_q W_r^{p q} y_{q h + s}.
// Afterwards lane j holds X[k + E rev(j)], k < E, where rev reverses the digits p of j. Inverse
// transforms conjugate every twiddle. lane_fft_adjoint applies the conjugate transpose of the whole
// sequence, which takes the digit-reversed distribution back to x[j + L n] and is the unnormalised
// inverse DFT: a forward transform, a pointwise product and the adjoint need no reordering in between.
//
// With radices 3 and 5 across lanes, the lengths with those factors need no shared-memory Stockham passes, whose
// nine barriers and run-time radices bound a slab stage (54 x 60 x 72, one evaluation of 23901 atoms at p = 5:
// influence stage 19.7 -> 6.3 us, slab stages 18.3 and 18.5 -> 13 us each under ncu, 50.0 -> 33.4 us in all).

// Unit u -> (transform t, lane j): warp u / 32 holds T = floor(32 / L) transforms at lane ids t mod T + T j. Lanes
// past the last transform get a t beyond any count: they work on a valid transform without storing.
template <int L>
PME_DEV void lane_unit(int u, int &t, int &j) {
    constexpr int T = 32 / L;
    const int lid = u & 31;
    t = (u >> 5) * T + (T * L == 32 ? lid & (T - 1) : lid % T);
    j = lid / T;
    if (T * L < 32 && j >= L) {
        t = 1 << 24;
        j = 0;
    }
}

// Units covering ntr transforms of L lanes: whole warps.
template <int L>
PME_DEV int lane_units(int ntr) {
    constexpr int T = 32 / L;
    return ((ntr + T - 1) / T) * 32;
}

PME_HD int lane_radix(int M) { return M % 5 == 0 ? 5 : (M % 3 == 0 ? 3 : 2); }
PME_HD int lane_rounds(int L) { return L <= 1 ? 0 : 1 + lane_rounds(L / lane_radix(L)); }

// Powers of two keep their own loops (bit operations and xor shuffles) below.
PME_HD bool lane_pow2(int L) { return (L & (L - 1)) == 0; }

template <int L, int M = L>
PME_DEV int lane_rev(int j) {
    if constexpr (lane_pow2(L)) {
        int r = 0;
#pragma unroll
        for (int b = 1; b < L; b <<= 1) r = (r << 1) | ((j & b) ? 1 : 0);
        return r;
    } else if constexpr (M <= 1) {
        return 0;
    } else {
        constexpr int r = lane_radix(M), h = M / r;
        const int p = (int)((unsigned)j / h);
        return p + r * lane_rev<L, h>(j - p * h);
    }
}

// The twiddles one lane needs (forward sign), loaded once so their latency overlaps the data loads and
// the inverse / adjoint transforms reuse them: w[k - 1] = W_N^{j k}, k = 1 .. E - 1, and for round i on groups
// of M lanes r[i] = W_M^{j mod h} (radix 2) or W_M^{p s} (radix 3, 5).
template <int L, int E>
struct LaneTw {
    float2 w[E > 1 ? E - 1 : 1];
    float2 r[lane_rounds(L) > 0 ? lane_rounds(L) : 1];
};

template <int L, int E, bool GLOBAL, int M, int I>
PME_DEV void lane_tw_rounds(const float2 *tw, int j, LaneTw<L, E> &t) {
    if constexpr (M > 1) {
        constexpr int r = lane_radix(M), h = M / r;
        const int jm = (int)((unsigned)j % M), p = (int)((unsigned)jm / h), s = jm - p * h;
        const int idx = (r == 2 ? s : p * s) * (L * E / M);
        t.r[I] = GLOBAL ? __ldg(tw + idx) : tw[idx];
        lane_tw_rounds<L, E, GLOBAL, h, I + 1>(tw, j, t);
    }
}

// tw[t] = exp(-2 pi i t / N), t < N, in global (read-only path) or shared memory.
template <int L, int E, bool GLOBAL>
PME_DEV LaneTw<L, E> lane_tw(const float2 *tw, int j) {
    LaneTw<L, E> t;
    if (L > 1) {
#pragma unroll
        for (int k = 1; k < E; ++k) t.w[k - 1] = GLOBAL ? __ldg(tw + j * k) : tw[j * k];
        if constexpr (lane_pow2(L)) {
#pragma unroll
            for (int i = 0, h = L / 2; h >= 1; ++i, h >>= 1) {
                const int idx = (j & (h - 1)) * (L * E / (2 * h));
                t.r[i] = GLOBAL ? __ldg(tw + idx) : tw[idx];
            }
        } else {
            lane_tw_rounds<L, E, GLOBAL, L, 0>(tw, j, t);
        }
    }
    return t;
}

PME_DEV float2 shfl_xor_c(float2 v, int mask) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, mask), __shfl_xor_sync(0xffffffffu, v.y, mask));
}
PME_DEV float2 shfl_c(float2 v, int lane) {
    return make_float2(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane));
}

PME_DEV float2 cmul_c(float2 a, float2 w, bool conj) { return conj ? cmul(a, cconj(w)) : cmul(a, w); }

// Output p of the radix-r DFT over the values of the lanes l0, l0 + step, ..., for every v[k].
template <int R, int E, bool INV>
PME_DEV void lane_dft(float2 (&v)[E], int l0, int step, int p) {
    static_assert(R == 3 || R == 5, "odd radices");
    if constexpr (R == 3) {
        // cos, sin of 2 pi p / 3
        const float c = p ? -0.5f : 1.0f, s = p == 0 ? 0.0f : (p == 1 ? 0.86602540378443864676f : -0.86602540378443864676f);
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const float2 a0 = shfl_c(v[k], l0), a1 = shfl_c(v[k], l0 + step), a2 = shfl_c(v[k], l0 + 2 * step);
            const float2 t = cadd(a1, a2), u = cmul_mi<INV>(csub(a1, a2));
            v[k] = make_float2(a0.x + c * t.x + s * u.x, a0.y + c * t.y + s * u.y);
        }
    } else {
        const float C1 = 0.30901699437494742410f, S1 = 0.95105651629515357212f;   // cos, sin of 2 pi / 5
        const float C2 = -0.80901699437494742410f, S2 = 0.58778525229247312917f;  // cos, sin of 4 pi / 5
        const float c1 = p == 0 ? 1.0f : (p == 1 || p == 4 ? C1 : C2), c2 = p == 0 ? 1.0f : (p == 1 || p == 4 ? C2 : C1);
        const float s1 = p == 0 ? 0.0f : (p == 1 ? S1 : (p == 2 ? S2 : (p == 3 ? -S2 : -S1)));
        const float s2 = p == 0 ? 0.0f : (p == 1 ? S2 : (p == 2 ? -S1 : (p == 3 ? S1 : -S2)));
#pragma unroll
        for (int k = 0; k < E; ++k) {
            const float2 a0 = shfl_c(v[k], l0), a1 = shfl_c(v[k], l0 + step), a2 = shfl_c(v[k], l0 + 2 * step),
                         a3 = shfl_c(v[k], l0 + 3 * step), a4 = shfl_c(v[k], l0 + 4 * step);
            const float2 t1 = cadd(a1, a4), t2 = cadd(a2, a3), u1 = cmul_mi<INV>(csub(a1, a4)), u2 = cmul_mi<INV>(csub(a2, a3));
            v[k] = make_float2(a0.x + c1 * t1.x + c2 * t2.x + s1 * u1.x + s2 * u2.x,
                               a0.y + c1 * t1.y + c2 * t2.y + s1 * u1.y + s2 * u2.y);
        }
    }
}

// The cross-lane rounds from groups of M lanes down, round I first.
template <int L, int E, bool INV, int M, int I>
PME_DEV void lane_rounds_down(float2 (&v)[E], int j, const LaneTw<L, E> &tw) {
    if constexpr (M > 1) {
        constexpr int T = 32 / L, r = lane_radix(M), h = M / r;
        if constexpr (r == 2) {
            const bool up = (unsigned)j % M >= (unsigned)h;
            const int other = (int)(threadIdx.x & 31) + (up ? -h : h) * T;
#pragma unroll
            for (int k = 0; k < E; ++k) {
                const float2 q = shfl_c(v[k], other);
                v[k] = up ? (h > 1 ? cmul_c(csub(q, v[k]), tw.r[I], INV) : csub(q, v[k])) : cadd(v[k], q);
            }
        } else {
            const int jm = (int)((unsigned)j % M), p = (int)((unsigned)jm / h);
            lane_dft<r, E, INV>(v, (int)(threadIdx.x & 31) - p * h * T, h * T, p);
            if (h > 1) {
#pragma unroll
                for (int k = 0; k < E; ++k) v[k] = cmul_c(v[k], tw.r[I], INV);
            }
        }
        lane_rounds_down<L, E, INV, h, I + 1>(v, j, tw);
    }
}

// Their conjugate transposes, the last round first.
template <int L, int E, int M, int I>
PME_DEV void lane_rounds_up(float2 (&v)[E], int j, const LaneTw<L, E> &tw) {
    if constexpr (M > 1) {
        constexpr int T = 32 / L, r = lane_radix(M), h = M / r;
        lane_rounds_up<L, E, h, I + 1>(v, j, tw);
        if constexpr (r == 2) {
            const bool up = (unsigned)j % M >= (unsigned)h;
            const int other = (int)(threadIdx.x & 31) + (up ? -h : h) * T;
            if (up && h > 1) {
#pragma unroll
                for (int k = 0; k < E; ++k) v[k] = cmul_c(v[k], tw.r[I], true);
            }
#pragma unroll
            for (int k = 0; k < E; ++k) {
                const float2 q = shfl_c(v[k], other);
                v[k] = up ? csub(q, v[k]) : cadd(v[k], q);
            }
        } else {
            const int jm = (int)((unsigned)j % M), p = (int)((unsigned)jm / h);
            if (h > 1) {
#pragma unroll
                for (int k = 0; k < E; ++k) v[k] = cmul_c(v[k], tw.r[I], true);
            }
            lane_dft<r, E, true>(v, (int)(threadIdx.x & 31) - p * h * T, h * T, p);
        }
    }
}

template <int L, int E, bool INV>
PME_DEV void lane_fft(float2 (&v)[E], int j, const LaneTw<L, E> &tw) {
    dft_small<E, INV>(v);
    if (L > 1) {
#pragma unroll
        for (int k = 1; k < E; ++k) v[k] = cmul_c(v[k], tw.w[k - 1], INV);
        if constexpr (lane_pow2(L)) {
            constexpr int T = 32 / L;
#pragma unroll
            for (int i = 0, h = L / 2; h >= 1; ++i, h >>= 1) {
                const bool up = (j & h) != 0;
#pragma unroll
                for (int k = 0; k < E; ++k) {
                    const float2 p = shfl_xor_c(v[k], h * T);
                    v[k] = up ? (h > 1 ? cmul_c(csub(p, v[k]), tw.r[i], INV) : csub(p, v[k])) : cadd(v[k], p);
                }
            }
        } else {
            lane_rounds_down<L, E, INV, L, 0>(v, j, tw);
        }
    }
}

template <int L, int E>
PME_DEV void lane_fft_adjoint(float2 (&v)[E], int j, const LaneTw<L, E> &tw) {
    if (L > 1) {
        if constexpr (lane_pow2(L)) {
            constexpr int T = 32 / L;
#pragma unroll
            for (int i = lane_rounds(L) - 1, h = 1; h < L; --i, h <<= 1) {
                const bool up = (j & h) != 0;
                if (up && h > 1) {
#pragma unroll
                    for (int k = 0; k < E; ++k) v[k] = cmul_c(v[k], tw.r[i], true);
                }
#pragma unroll
                for (int k = 0; k < E; ++k) {
                    const float2 p = shfl_xor_c(v[k], h * T);
                    v[k] = up ? csub(p, v[k]) : cadd(v[k], p);
                }
            }
        } else {
            lane_rounds_up<L, E, L, 0>(v, j, tw);
        }
#pragma unroll
        for (int k = 1; k < E; ++k) v[k] = cmul_c(v[k], tw.w[k - 1], true);
    }
    dft_small<E, true>(v);
}
#endif  // warps

}  // namespace pme
