// Site-local fifth-dimension operators: out = coef * Op in (+ x), Op one of
// the s-operators of each chirality (I^-1 by the closed-form elimination of
// Sec. 3, M_phi, K = M_phi I^-1, the shift C, or a dense Ls x Ls table), or
// their adjoints (chirality swapped). The Ls spinors of a 4d site are staged
// in shared memory and each (site, component) column is solved by one thread.
#include "fx.cuh"
#include "mdwf_internal.cuh"

namespace mdwf {

// the result in its field, or in fixed point for the FP64 hops that read it
template <int P, typename R>
__device__ __forceinline__ void store_m5(const Field<P>& f, int* exp, long long sr, int s, const R* v) {
    if constexpr (P == MDWF_F64) {
        if (exp) {
            fx_store(f, exp, sr, s, v);
            return;
        }
    }
    f.store(sr, s, v);
}

// FORM: the operators that read a spinor and its two neighbours straight from memory (below), whole columns in
// shared memory, or dense tables: kernels of their own, since in one the registers of each form held the others back.
// Blocks per SM: FP32 and FP16+norm eight (64 registers; at 75 and six blocks M_phi of 16^3 x 32 x 16 took 31.0 and
// 26.6 us, now 30.5 and 24.5). FP64 direct four, 72 us (six in one kernel: 105); FP64 columns, which wait for the FP64
// pipe and for each other, six: A^dag 142 us at 78 registers (one kernel with four blocks, 120 registers: 176); FP64
// dense four.
enum { M5_DIRECT, M5_COLUMNS, M5_DENSE };
template <int P, bool XPAY, int FORM>
__global__ void __launch_bounds__(128, P != MDWF_F64 ? 8 : FORM == M5_COLUMNS ? 6 : 4)
    m5_kernel(Field<P> out, Field<P> in, Field<P> xf, const typename PrecTraits<P>::real* tab,
              const typename PrecTraits<P>::real* mass, typename PrecTraits<P>::real coef, Geom g, int sop, int swap,
              SCoef<typename PrecTraits<P>::real> sc, const double* mask, int* out_exp) {
    typedef typename PrecTraits<P>::real R;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Ls = g.Ls;
    constexpr bool dense = FORM == M5_DENSE;
    R* mat = reinterpret_cast<R*>(smem_raw);
    R* cs = mat + (dense ? 2 * Ls * Ls : 0);
    const int nrhs = (int)(gridDim.x / ((g.Vh + blockDim.y - 1) / blockDim.y));
    const int s = threadIdx.x, ly = threadIdx.y, rhs = blockIdx.x % nrhs;
    if (mask && mask[rhs] == 0.0) return;  // block-uniform, before any barrier
    const long long sblk = blockIdx.x / nrhs;
    const int tid = ly * blockDim.x + s, nthr = blockDim.x * blockDim.y;
    // The bidiagonal operators (M_phi, C, I = M+ + M- C) and the identity need only
    // the s +- 1 neighbours of a column, which share the thread's cache lines: each
    // thread reads its spinor and the two half spinors straight from memory, with no
    // staging and no barrier (the identity also in place; the others out of place,
    // since a neighbour's element may be overwritten). Chirality 0 (reals 0..11)
    // couples to s - 1 and chirality 1 to s + 1; the adjoint (swap) exchanges them;
    // the wrap-around term carries -m. Block-uniform.
    if constexpr (FORM == M5_DIRECT) {
        const long long site = sblk * blockDim.y + ly;
        if (site >= g.Vh) return;
        const long long sr = (long long)rhs * g.Vh + site;
        R v[24];
        in.load(sr, s, v);
        if (sop != SOP_ID) {
            R w0, w1;
            bidiag_weights(sop, sc, w0, w1);
            const R m = mass[rhs];
            const bool sw = swap != 0;
            const int up = s + 1 < Ls ? s + 1 : 0, dn = s > 0 ? s - 1 : Ls - 1;
            const R f0 = w1 * ((sw ? s < Ls - 1 : s > 0) ? R(1) : -m);
            const R f1 = w1 * ((sw ? s > 0 : s < Ls - 1) ? R(1) : -m);
            R h0[12], h1[12];
            in.load_half(sr, sw ? up : dn, 0, h0);
            in.load_half(sr, sw ? dn : up, 1, h1);
            // FP64: no product with w0 = 1 (2 FP64 operations a clock and SM); the others: no second branch (registers)
            if (P != MDWF_F64 || w0 != R(1)) {
#pragma unroll
                for (int k = 0; k < 24; ++k) v[k] *= w0;
            }
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                v[k] = fma(f0, h0[k], v[k]);
                v[12 + k] = fma(f1, h1[k], v[12 + k]);
            }
        }
        if (XPAY) {
            R xv[24];
            xf.load(sr, s, xv);
#pragma unroll
            for (int k = 0; k < 24; ++k) v[k] = fma(coef, v[k], xv[k]);
        } else if (coef != R(1)) {
#pragma unroll
            for (int k = 0; k < 24; ++k) v[k] *= coef;
        }
        store_m5(out, out_exp, sr, s, v);
        return;
    }
    if (dense) {
        const R* gm = tab + (size_t)rhs * 2 * Ls * Ls;
        for (int i = tid; i < 2 * Ls * Ls; i += nthr) mat[i] = gm[i];
    }
    const long long site = sblk * blockDim.y + ly;
    const bool active = site < g.Vh;
    const long long sr = (long long)rhs * g.Vh + site;
    R v[24];
    if (active) in.load(sr, s, v);
    else {
#pragma unroll
        for (int k = 0; k < 24; ++k) v[k] = 0;
    }
    const int sst = site_stride(Ls);
    R* mine = cs + (size_t)ly * sst + s * kRowStride;
    row_store(mine, v);
    __syncthreads();
    R res[24];
    if (dense) {
        if (!active) return;
#pragma unroll
        for (int k = 0; k < 24; ++k) res[k] = 0;
        const R* col = cs + (size_t)ly * sst;
        for (int sp = 0; sp < Ls; ++sp) {
            const R mp = mat[sp * Ls + s], mm = mat[(Ls + sp) * Ls + s];
            const R* h = col + sp * kRowStride;
#pragma unroll
            for (int k = 0; k < 12; ++k) res[k] += mp * h[k];
#pragma unroll
            for (int k = 12; k < 24; ++k) res[k] += mm * h[k];
        }
    } else {
        // the shared-memory walk: register-held columns measured slower in this kernel
        const SMass<R> sm{mass[rhs], mass[kMaxRhs + rhs]};
        block_columns(cs, blockDim.y, Ls, sop, swap != 0, sc, sm, tid, nthr, false);
        __syncthreads();
        if (!active) return;
        row_load(mine, res);
    }
    if (XPAY) {
        R xv[24];
        xf.load(sr, s, xv);
#pragma unroll
        for (int k = 0; k < 24; ++k) res[k] = fma(coef, res[k], xv[k]);
    } else if (coef != R(1)) {
#pragma unroll
        for (int k = 0; k < 24; ++k) res[k] *= coef;
    }
    store_m5(out, out_exp, sr, s, res);
}

template <int P>
static int launch_m5_t(mdwf_ctx* c, const M5Launch& m) {
    typedef typename PrecTraits<P>::real R;
    const Geom& g = c->g;
    int SB = 128 / g.Ls;
    if (SB < 1) SB = 1;
    dim3 block(g.Ls, SB), grid((unsigned)((g.Vh + SB - 1) / SB * m.nrhs));  // rhs fastest
    size_t smem = (size_t)((m.sop == SOP_DENSE ? 2 * g.Ls * g.Ls : 0) + SB * site_stride(g.Ls)) * sizeof(R);
    Field<P> out = make_field<P>(m.out, g, m.nrhs);
    Field<P> in = make_field<P>(const_cast<void*>(m.in), g, m.nrhs);
    Field<P> xf = m.x ? make_field<P>(const_cast<void*>(m.x), g, m.nrhs) : out;
    const R* tab = reinterpret_cast<const R*>(m.mat);
    const R* mass = m.mass ? reinterpret_cast<const R*>(m.mass)
                           : P == MDWF_F64 ? reinterpret_cast<const R*>(c->mass64)
                                           : reinterpret_cast<const R*>(c->mass32);
    const SCoef<R> sc = make_scoef<R>(c);
    const R coef = (R)(m.unscaled ? m.coef : m.coef * sop_scale(c, m.sop));
    const double n5 = (double)g.Vh * g.Ls * m.nrhs;
    LaunchScope scope(c, (m.x ? KB_M5_XPAY : KB_M5) * 3 + P, n5 * site_bytes(P) * (m.x ? 3.0 : 2.0),
                      n5 * (144.0 + (m.x ? 24.0 : 0.0)));
    auto launch = [&](auto k) {
        if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k<<<grid, block, smem, c->stream>>>(out, in, xf, tab, mass, coef, g, m.sop, m.swap, sc, m.mask, m.out_exp);
    };
    const bool bidiag = m.sop == SOP_MPHI || m.sop == SOP_C || m.sop == SOP_MEE;
    if (m.sop == SOP_DENSE)
        m.x ? launch(m5_kernel<P, true, M5_DENSE>) : launch(m5_kernel<P, false, M5_DENSE>);
    else if (m.sop == SOP_ID || (bidiag && m.out != m.in))
        m.x ? launch(m5_kernel<P, true, M5_DIRECT>) : launch(m5_kernel<P, false, M5_DIRECT>);
    else
        m.x ? launch(m5_kernel<P, true, M5_COLUMNS>) : launch(m5_kernel<P, false, M5_COLUMNS>);
    return check_launch();
}

int launch_m5(mdwf_ctx* c, int prec, const M5Launch& m) {
    switch (prec) {
        case MDWF_F64: return launch_m5_t<MDWF_F64>(c, m);
        case MDWF_F32: return launch_m5_t<MDWF_F32>(c, m);
        case MDWF_F16N: return launch_m5_t<MDWF_F16N>(c, m);
    }
    return MDWF_EINVAL;
}

}  // namespace mdwf
