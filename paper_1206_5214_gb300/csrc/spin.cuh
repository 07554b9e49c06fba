// Spin projection, colour transport and reconstruction of one Wilson hopping term.
#pragma once

#include <cuda_runtime.h>

namespace mdwf {

// --------------------------------------------------------- spin structure
//
// Chiral basis g_mu = [[0, A_mu], [A_mu^dag, 0]], A_k = -i sigma_k, A_4 = 1.
// (1 + S g_mu) psi, psi = (u, l) by chirality halves, has upper half
// h = u + S A l and lower half S A^dag h, so only h (2 spins x 3 colours) is
// transported: project -> multiply by the link -> reconstruct.

template <int MU, int S, typename R>
__device__ __forceinline__ void project(const R* w, R* h) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R u0r = w[2 * c], u0i = w[2 * c + 1], u1r = w[6 + 2 * c], u1i = w[7 + 2 * c];
        const R l0r = w[12 + 2 * c], l0i = w[13 + 2 * c], l1r = w[18 + 2 * c], l1i = w[19 + 2 * c];
        R a0r, a0i, a1r, a1i;  // (A l)_0, (A l)_1
        if (MU == 0) {         // A = -i sigma_1: (A l)_0 = -i l1, (A l)_1 = -i l0
            a0r = l1i; a0i = -l1r; a1r = l0i; a1i = -l0r;
        } else if (MU == 1) {  // A = -i sigma_2: (A l)_0 = -l1, (A l)_1 = l0
            a0r = -l1r; a0i = -l1i; a1r = l0r; a1i = l0i;
        } else if (MU == 2) {  // A = -i sigma_3: (A l)_0 = -i l0, (A l)_1 = i l1
            a0r = l0i; a0i = -l0r; a1r = -l1i; a1i = l1r;
        } else {               // A = 1
            a0r = l0r; a0i = l0i; a1r = l1r; a1i = l1i;
        }
        h[2 * c] = u0r + S * a0r;
        h[2 * c + 1] = u0i + S * a0i;
        h[6 + 2 * c] = u1r + S * a1r;
        h[7 + 2 * c] = u1i + S * a1i;
    }
}

// Colour i of a transported half spinor g (2 spins, re and im): the upper half of (1 + S g_mu) gets g,
// the lower half S A_mu^dag g.
template <int MU, int S, typename R>
__device__ __forceinline__ void reconstruct_colour(R* acc, int i, const R* g) {
    const R g0r = g[0], g0i = g[1], g1r = g[2], g1i = g[3];
    acc[2 * i] += g0r;
    acc[2 * i + 1] += g0i;
    acc[6 + 2 * i] += g1r;
    acc[7 + 2 * i] += g1i;
    R b0r, b0i, b1r, b1i;  // (A^dag g)_0, (A^dag g)_1
    if (MU == 0) {         // A^dag = i sigma_1: (i g1, i g0)
        b0r = -g1i; b0i = g1r; b1r = -g0i; b1i = g0r;
    } else if (MU == 1) {  // A^dag = i sigma_2: (g1, -g0)
        b0r = g1r; b0i = g1i; b1r = -g0r; b1i = -g0i;
    } else if (MU == 2) {  // A^dag = i sigma_3: (i g0, -i g1)
        b0r = -g0i; b0i = g0r; b1r = g1i; b1i = -g1r;
    } else {
        b0r = g0r; b0i = g0i; b1r = g1r; b1i = g1i;
    }
    acc[12 + 2 * i] += S * b0r;
    acc[13 + 2 * i] += S * b0i;
    acc[18 + 2 * i] += S * b1r;
    acc[19 + 2 * i] += S * b1i;
}

// Transport and reconstruction of one hopping term: g[a][i] = sum_j V[i][j] h[a][j]
// with V = U (or U^dag when ADJ; U row-major complex 3x3), then the upper half
// of (1 + S g_mu) gets g and the lower half S A_mu^dag g. It runs one output
// colour i at a time so that only one colour of g is live; `scaled` multiplies
// g by `scale` first (the FP16 norm of the neighbour).
template <bool ADJ, int MU, int S, typename R>
__device__ __forceinline__ void transport_add(R* acc, const R* U, const R* h, R scale, bool scaled) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        R g[4];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            // complex multiply-accumulate as four fused multiply-adds per term
            R sr = 0, si = 0;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const R ur = ADJ ? U[2 * (3 * j + i)] : U[2 * (3 * i + j)];
                const R ui = ADJ ? -U[2 * (3 * j + i) + 1] : U[2 * (3 * i + j) + 1];
                const R hr = h[6 * a + 2 * j], hi = h[6 * a + 2 * j + 1];
                sr = fma(ur, hr, sr);
                sr = fma(-ui, hi, sr);
                si = fma(ur, hi, si);
                si = fma(ui, hr, si);
            }
            g[2 * a] = scaled ? scale * sr : sr;
            g[2 * a + 1] = scaled ? scale * si : si;
        }
        reconstruct_colour<MU, S>(acc, i, g);
    }
}

// Reconstruction alone, for a half spinor g already transported (the backward
// t-direction term of a slab face, whose link lives on the sending slab):
// upper half += f g, lower half += f S A_mu^dag g.
template <int MU, int S, typename R>
__device__ __forceinline__ void reconstruct_add(R* acc, const R* g, R f) {
    static_assert(MU == 3, "slab faces are t-faces (A_4 = 1)");
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        acc[k] = fma(f, g[k], acc[k]);
        acc[12 + k] = fma(S * f, g[k], acc[12 + k]);
    }
}

}  // namespace mdwf
