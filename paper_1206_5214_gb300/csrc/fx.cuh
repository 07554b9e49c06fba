// Fixed-point form of the FP64 hopping operator's operands, and the hopping sum on it.
//
// Why: GB300 issues 2 FP64 FMAs per clock and SM (measured 2.1), but 32 products of two 32-bit integers with a
// 64-bit result and 64 64-bit integer additions (the compiler makes one of each from a multiply-add). The hopping
// sum of one 5d site is about 770 FP64 operations, which bound the FP64 operator at 1.8 ms per hop on 16^3 x 32 x
// 16 with the memory nearly idle. On 64-bit integers it is 1728 products and additions of 32-bit limbs and some
// thousand cheap operations: 0.44 to 0.49 ms per hop with the s-operator of the epilogue, M 3.82 -> 1.01 ms, M^dag
// 3.92 -> 1.06 ms. What bounds it now: about 8000 instructions per 5d site at 16 warps per SM (128 registers),
// issued on 42 % of the cycles; the multiplier is 54 % busy, the FP64 pipe (s-operators) 32 %. One integer product
// of the upper parts with FP32 cross terms needs a third of the products and was 5 % faster, but its error was
// above that of FP64 in a quarter of the cases.
//
// Format: the 24 reals of one (site, s) spinor share a binary exponent e (the largest biased exponent among them)
// and are stored as signed 64-bit integers q with value q 2^(e - 1080), |q| < 2^58. A link's 18 reals share one in
// the same way, value u 2^(e - 1083), |u| < 2^61; they are stored as two signed 32-bit limbs, u = hi 2^32 + lo.
//
// Error: a product drops lo x lo (below 2^62, a quarter of the last place of the sum) and the sum of a term's six
// products is rounded to a multiple of 2^64, so a hopping sum is off by about one unit where the largest of its
// eight neighbours' components, times a link entry of one, is 2^54 to 2^55 units. FP64 arithmetic rounds every
// partial sum to 2^-53 of its size. M and M^dag against long double, 24 cases of lattices, Ls, links and
// coefficients and four kinds of input (Gaussian, slices falling by e^-2, point source, sites spread over decades):
// mean relative error 1.62e-16 with FP64 hops, 1.18e-16 with these and today's s-operators; per site as well.
// Ranges: a neighbour's projected component is below 2^59 (limbs |hi| <= 2^27, |lo| <= 2^31), so the middle sum is
// at most 6 (2^29 2^31 + 2^31 2^27) = 7.5 2^60 < 2^63, a transported component at most 6 2^56, and the sum of eight
// terms at most 48 2^56 < 2^63.
//
// Small parts beside large ones: the error above is relative to the largest component that reaches a site, where
// FP64 arithmetic errs relative to what each component is made of. The two differ where parts of the field do not
// mix: a hopping term adds to an upper spin only that spin and the lower ones (and the reverse), and links diagonal
// in colour (a free field) keep the colours apart. So a spinor is stored in fixed point only if in every colour
// each spin, together with the two of the other chirality, reaches 2^-kFxSpread of the largest component, and a
// link only if its rows and columns do; others (point sources, fields of one colour) are kept as raw doubles. The
// terms of a component then add up to 2^(54 - kFxSpread) units times a link entry (0.57 in the row of a unitary
// link), 2^45, or more. The eight terms are off by 25 units at most (each: 0.9 for the truncated fields, 0.2 for
// the links, 1.5 for lo x lo, 0.5 for the rounding) and by 1.5 in the root mean square: 7e-13 and 4e-14 of the
// component's terms at the very edge of the rule, FP64's accuracy away from it. Gaussian fields cross the line at
// one spinor in 10^11. Fields of one chirality alone, such as the sources of four-dimensional quarks, cross it at
// one in 2700, and a warp reads 256: M on 16^3 x 32 x 16 then takes 1.39 ms, 2.2 for one colour, 1.01 otherwise
// (1.006 without the rule; 3.8 in FP64 arithmetic). With kFxSpread = 7 one chirality takes 2.26 ms, with 5 it takes
// 3.4 and the FP64 solve on 8^3 x 16 x 12 79 instead of 64.6; with 10 it takes 1.07, but the bound passes 1e-12. In
// the solves the chiralities stay within a factor of 1.2 of each other.
//
// Raw spinors and links carry the exponent kFxRaw, and a site that has such a neighbour (or link) takes the FP64
// arithmetic; non-finite ones are stored so too, so that infinities and NaN spread as there.
#pragma once

#include "mdwf_internal.cuh"

namespace mdwf {

constexpr int kFxFieldBias = 1080, kFxLinkBias = 1083;
constexpr int kFxZero = -(1 << 20);   // exponent of an all-zero spinor or link
constexpr int kFxRaw = 1 << 24;       // exponent of a spinor or link kept as doubles
constexpr int kFxRawMin = 1 << 22;    // sums of exponents at or above this hold a kFxRaw
constexpr int kFxSpread = 8;          // binary orders between the parts of a fixed-point spinor or link

// the upper word of |v|: sizes compare by it to a tenth of a binary order
__device__ __forceinline__ int fx_size(double v) { return __double2hiint(v) & 0x7fffffff; }

// the exponent of a spinor; kFxRaw where its parts are too far apart for one (the rule above, zero parts included)
__device__ __forceinline__ int fx_spinor_exponent(const double* v) {
    int top = 0, low = 0x7fffffff, rest = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int a[4];  // the four spins
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const double re = v[6 * b + 2 * c], im = v[6 * b + 2 * c + 1];
            a[b] = max(fx_size(re), fx_size(im));
            rest |= __double2loint(re) | __double2loint(im);
        }
        const int u = max(a[0], a[1]), l = max(a[2], a[3]);
        low = min(low, min(max(min(a[0], a[1]), l), max(min(a[2], a[3]), u)));
        top = max(top, max(u, l));
    }
    if ((top | rest) == 0) return kFxZero;
    if ((top >> 20) == 0x7ff || low < top - (kFxSpread << 20)) return kFxRaw;
    return max(top >> 20, 1);  // subnormals carry the exponent 1
}

// the exponent of a link, by its rows and columns
__device__ __forceinline__ int fx_link_exponent(const double* v) {
    int row[3] = {0, 0, 0}, col[3] = {0, 0, 0}, rest = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int a = max(fx_size(v[2 * k]), fx_size(v[2 * k + 1]));
        row[k / 3] = max(row[k / 3], a);
        col[k % 3] = max(col[k % 3], a);
        rest |= __double2loint(v[2 * k]) | __double2loint(v[2 * k + 1]);
    }
    const int top = max(row[0], max(row[1], row[2]));
    const int low = min(min(row[0], min(row[1], row[2])), min(col[0], min(col[1], col[2])));
    if ((top | rest) == 0) return kFxZero;
    if ((top >> 20) == 0x7ff || low < top - (kFxSpread << 20)) return kFxRaw;
    return max(top >> 20, 1);
}

// v as an integer at the shared exponent e, with SH guard bits below the 53 of a double (truncated)
template <int SH>
__device__ __forceinline__ long long fx_mantissa(double v, int e) {
    const int hi = __double2hiint(v);
    const int ev = (hi >> 20) & 0x7ff;
    const unsigned mh = (unsigned)(hi & 0xfffff) | (ev ? 0x100000u : 0u);
    unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)__double2loint(v)) << SH;
    m >>= min(e - max(ev, 1), 63);
    return hi < 0 ? -(long long)m : (long long)m;
}

__device__ __forceinline__ void fx_split(long long v, int& hi, int& lo) {
    lo = (int)v;
    hi = (int)((v + 0x80000000ll) >> 32);
}

// a 2^x as a double, rounded to nearest, by integer operations (the FP64 pipe would take a conversion and
// a multiplication); x must keep the result a normal number (fx_scale_safe)
__device__ __forceinline__ double fx_to_double(long long a, int x) {
    const long long sgn = a >> 63;
    const unsigned long long m0 = (unsigned long long)((a ^ sgn) - sgn);
    const int lz = __clzll((long long)m0);
    const unsigned long long m = m0 << (lz & 63);               // the top bit at 63
    const unsigned long long rr = (m >> 11) + ((m >> 10) & 1);  // 53 bits, or 2^53 after a carry
    const unsigned long long bits = ((unsigned long long)(unsigned)(1085 - lz + x) << 52) + rr;
    const double d = __longlong_as_double((long long)(bits | ((unsigned long long)sgn << 63)));
    return m0 == 0 ? 0.0 : d;
}
__device__ __forceinline__ bool fx_scale_safe(int x) { return x >= -1000 && x <= 950; }

// Device view of a fixed-point field: the FP64 field's layout with integers, and [rhs][site][s] exponents.
struct FxField {
    const longlong2* v;
    const int* e;
    int Ls;
    Bounds bnd;
    __device__ __forceinline__ int exponent(long long sr, int s) const {
        if (bnd.bad(sr, s, Ls)) return kFxZero;
        return __ldg(e + sr * Ls + s);
    }
    __device__ __forceinline__ void load(long long sr, int s, long long* o) const {
        if (bnd.bad(sr, s, Ls)) { for (int k = 0; k < 24; ++k) o[k] = 0; return; }
        const longlong2* p = v + sr * 12 * Ls + s;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const longlong2 d = __ldg(p + (long long)k * Ls);
            o[2 * k] = d.x;
            o[2 * k + 1] = d.y;
        }
    }
    // the spinor as doubles, exactly (the path of raw neighbours)
    __device__ __forceinline__ void load(long long sr, int s, double* o) const {
        long long q[24];
        load(sr, s, q);
        const int e = exponent(sr, s), x = e - kFxFieldBias;
        if (e == kFxRaw) {
#pragma unroll
            for (int k = 0; k < 24; ++k) o[k] = __longlong_as_double(q[k]);
        } else if (fx_scale_safe(x)) {
#pragma unroll
            for (int k = 0; k < 24; ++k) o[k] = fx_to_double(q[k], x);
        } else {
            for (int k = 0; k < 24; ++k) o[k] = e == kFxZero ? 0.0 : scalbn((double)q[k], x);
        }
    }
};

// writes a spinor of doubles in fixed point
__device__ __forceinline__ void fx_store(const Field<MDWF_F64>& f, int* e, long long sr, int s, const double* v) {
    if (f.bnd.bad(sr, s, f.Ls)) return;
    const int x = fx_spinor_exponent(v);
    longlong2* p = reinterpret_cast<longlong2*>(f.v) + sr * 12 * f.Ls + s;
    if (x == kFxRaw) {
#pragma unroll
        for (int k = 0; k < 12; ++k)
            p[(long long)k * f.Ls] = make_longlong2(__double_as_longlong(v[2 * k]), __double_as_longlong(v[2 * k + 1]));
    } else {
#pragma unroll
        for (int k = 0; k < 12; ++k)
            p[(long long)k * f.Ls] = make_longlong2(fx_mantissa<5>(v[2 * k], x), fx_mantissa<5>(v[2 * k + 1], x));
    }
    e[sr * f.Ls + s] = x;
}

// Fixed-point links: [link][9] of (re lo, re hi, im lo, im hi), and one exponent per link. A context without
// them has the exponents alone, all kFxRaw.
struct FxGauge {
    const int4* u;
    const int* e;
    Bounds bnd;
};

}  // namespace mdwf
