// The hopping sum of the FP64 operator on fixed-point fields and links (the format, its error and why it
// pays: fx.cuh).
#pragma once

#include "fx.cuh"
#include "spin.cuh"

namespace mdwf {

// (v f) 2^-62 for a factor f below 2^62
__device__ __forceinline__ long long fx_scale(long long v, long long f) {
    const long long hi = __mul64hi(v, f);
    const unsigned long long lo = (unsigned long long)v * (unsigned long long)f;
    return (long long)(((unsigned long long)hi << 2) | (lo >> 62));
}

// a b + c, 32 x 32 + 64 bits. Written out: where the compiler sees that a limb is the upper half of a 64-bit
// value it multiplies 64-bit operands, which takes several times the instructions.
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// The colour product g[a][i] = sum_j V_ij h[a][j] on integers, V_ij = u[i si + j sj] (the link, or its transpose).
__device__ __forceinline__ void fx_colour(const int4* u, int si, int sj, const long long* h, long long* g) {
    int hh[12], hl[12], nh[6], nl[6];  // limbs; of the negated imaginary parts
#pragma unroll
    for (int k = 0; k < 12; ++k) fx_split(h[k], hh[k], hl[k]);
#pragma unroll
    for (int k = 0; k < 6; ++k) fx_split(-h[2 * k + 1], nh[k], nl[k]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        int4 r[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) r[j] = __ldg(u + i * si + j * sj);
        const long long half = 0x80000000ll;  // half of the place that is kept
        // four sums (2 spins, re and im) side by side, since one sum's multiply-adds depend on each other (two at a
        // time: M 1.021 against 1.004 ms; the upper parts beside them: 1.052, registers)
        long long m[4] = {half, half, half, half};
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    const int k = 6 * a + 2 * j, n = 3 * a + j;
                    const int u = p == 0 ? r[j].y : p == 1 ? r[j].x : p == 2 ? r[j].w : r[j].z;
                    m[2 * a] = mad_wide(u, p == 0 ? hl[k] : p == 1 ? hh[k] : p == 2 ? nl[n] : nh[n], m[2 * a]);
                    m[2 * a + 1] =
                        mad_wide(u, p == 0 ? hl[k + 1] : p == 1 ? hh[k + 1] : p == 2 ? hl[k] : hh[k], m[2 * a + 1]);
                }
#pragma unroll
        for (int k = 0; k < 4; ++k) m[k] >>= 32;
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const int k = 6 * a + 2 * j, n = 3 * a + j;
                m[2 * a] = mad_wide(r[j].y, hh[k], m[2 * a]);
                m[2 * a + 1] = mad_wide(r[j].y, hh[k + 1], m[2 * a + 1]);
                m[2 * a] = mad_wide(r[j].w, nh[n], m[2 * a]);
                m[2 * a + 1] = mad_wide(r[j].w, hh[k], m[2 * a + 1]);
            }
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            g[6 * a + 2 * i] = m[2 * a];
            g[6 * a + 2 * i + 1] = m[2 * a + 1];
        }
    }
}

// The spin parts of term (MU, FWD): the projected half spinor, and what the transported one adds to the sum. The
// backward term's colour product is with U^dag: (U^dag h) = conj(U^T conj(h)), so h and g are conjugated here and
// fx_colour takes the transpose.
template <int MU, int S, bool CONJ>
__device__ __forceinline__ void fx_project(const long long* w, long long* h) {
    project<MU, S>(w, h);
    if (CONJ) {
#pragma unroll
        for (int k = 1; k < 12; k += 2) h[k] = -h[k];
    }
}
template <int MU, int S, bool CONJ>
__device__ __forceinline__ void fx_reconstruct(long long* acc, const long long* g) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const long long c[4] = {g[2 * i], CONJ ? -g[2 * i + 1] : g[2 * i + 1], g[6 + 2 * i],
                                CONJ ? -g[7 + 2 * i] : g[7 + 2 * i]};
        reconstruct_colour<MU, S>(acc, i, c);
    }
}

// What the fixed-point hop needs beside the field views.
struct FxHop {
    FxField in;
    FxGauge U;
    int* out_exp;          // exponents of a fixed-point output, or null (FP64 output)
    long long ff, fb;      // time-term factors e^{+-mu} over 2^(62 + their exponent), 0: none
    int xf, xb;            // their exponents
};

// Terms t0, t0 + DT, ... of the eight of one (site, s), t = 0..3 the forward ones, 4..7 the backward ones: their sum
// as integers at the exponent `top` of the largest term of all eight. False where a neighbour or a link is
// raw (the caller then takes the FP64 arithmetic).
template <bool DAG, int DT>
__device__ __forceinline__ bool fx_terms(long long* acc, int& top, int t0, const FxHop& fx, const Geom& g,
                                         int out_parity, const int* nbi, long long site, int s, long long rbase) {
    constexpr int SF = DAG ? +1 : -1;
    // the exponent of term t, t = 0..3 the forward terms, 4..7 the backward ones
    auto term_exponent = [&](int t, long long j, long long l) {
        int e = fx.in.exponent(rbase + j, s);
        if (!fx.U.bnd.bad(l, 0, 1)) e += __ldg(fx.U.e + l);
        return t == 3 ? e + fx.xf : t == 7 ? e + fx.xb : e;
    };
    auto link_of = [&](int t, long long j) {
        return ((long long)(t < 4 ? out_parity : 1 - out_parity) * 4 + (t & 3)) * g.Vh + (t < 4 ? site : j);
    };
    top = kFxZero * 4;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const long long j = __ldg(nbi + t);
        top = max(top, term_exponent(t, j, link_of(t, j)));
    }
    if (top >= kFxRawMin) return false;
    // One body for the eight terms (the spin parts by uniform branches): unrolled, the compiler moves the loads of
    // later terms up and spills.
#pragma unroll 1
    for (int t = t0; t < 8; t += DT) {
        const long long j = __ldg(nbi + t), l = link_of(t, j);
        const int sh = min(top - term_exponent(t, j, l), 63);
        long long h[12], gg[12];
        {
            long long w[24];
            fx.in.load(rbase + j, s, w);
            switch (t) {
                case 0: fx_project<0, SF, false>(w, h); break;
                case 1: fx_project<1, SF, false>(w, h); break;
                case 2: fx_project<2, SF, false>(w, h); break;
                case 3: fx_project<3, SF, false>(w, h); break;
                case 4: fx_project<0, -SF, true>(w, h); break;
                case 5: fx_project<1, -SF, true>(w, h); break;
                case 6: fx_project<2, -SF, true>(w, h); break;
                default: fx_project<3, -SF, true>(w, h);
            }
        }
#pragma unroll
        for (int k = 0; k < 12; ++k) h[k] >>= sh;
        if (fx.U.bnd.bad(l, 0, 1)) continue;
        fx_colour(fx.U.u + l * 9, t < 4 ? 3 : 1, t < 4 ? 1 : 3, h, gg);
        if ((t & 3) == 3 && fx.ff) {
            const long long f = t < 4 ? fx.ff : fx.fb;
#pragma unroll
            for (int k = 0; k < 12; ++k) gg[k] = fx_scale(gg[k], f);
        }
        switch (t) {
            case 0: fx_reconstruct<0, SF, false>(acc, gg); break;
            case 1: fx_reconstruct<1, SF, false>(acc, gg); break;
            case 2: fx_reconstruct<2, SF, false>(acc, gg); break;
            case 3: fx_reconstruct<3, SF, false>(acc, gg); break;
            case 4: fx_reconstruct<0, -SF, true>(acc, gg); break;
            case 5: fx_reconstruct<1, -SF, true>(acc, gg); break;
            case 6: fx_reconstruct<2, -SF, true>(acc, gg); break;
            default: fx_reconstruct<3, -SF, true>(acc, gg);
        }
    }
    return true;
}

// The sum of the eight terms as doubles.
__device__ __forceinline__ void fx_finish(double* out, const long long* acc, int top) {
    // one unit of acc is 2^64 2^(e - kFxFieldBias) 2^(e' - kFxLinkBias), e + e' = top
    const int x = top - kFxFieldBias - kFxLinkBias + 64;
    if (fx_scale_safe(x)) {
#pragma unroll
        for (int k = 0; k < 24; ++k) out[k] = fx_to_double(acc[k], x);
    } else {  // results that are subnormal or overflow: 2^x in two factors
        const int y = min(max(x, -2140), 2000), half = y / 2;
        const double f1 = scalbn(1.0, half), f2 = scalbn(1.0, y - half);
#pragma unroll
        for (int k = 0; k < 24; ++k) out[k] = fx_to_double(acc[k], 0) * f1 * f2;
    }
}

}  // namespace mdwf
