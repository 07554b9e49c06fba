// Conversions between the user formats (complex128, lexicographic) and the
// internal per-parity, s-innermost layouts of every precision.
#include "fx.cuh"
#include "mdwf_internal.cuh"

namespace mdwf {

// User fields <-> internal fields. FULL: the user field is [rhs][s][2 Vh sites][24] and its sites alternate between
// the two parities (internal site = lexicographic index / 2); else it is [rhs][s][Vh odd sites][24] (odd only).
// A block takes SB consecutive user sites and their Ls slices: for each slice the user field holds SB 192 contiguous
// bytes, read (or written) with consecutive 16-byte accesses, and the internal field is accessed by its own chunks;
// shared memory turns one into the other. (One thread per (site, s) that walks its 192 bytes in the user field,
// with the slices of a site far apart, moved 1.8 TB/s: import and export of 16^3 x 32 x 16 FP32 took 341 us, now
// 133 us, 4.5 TB/s.)
// Rows of 13 double2 put the 16-byte row accesses of 8 consecutive threads on distinct banks.
constexpr int kLayoutRow = 13;

template <int P, bool FULL, bool TO_INTERNAL>
__global__ void __launch_bounds__(128) layout_kernel(Field<P> even, Field<P> odd, double* user, Geom g, int nrhs) {
    typedef typename PrecTraits<P>::real R;
    extern __shared__ __align__(16) double2 tile[];  // [site of the block][s][kLayoutRow]
    const int Ls = g.Ls, SB = blockDim.y, s = threadIdx.x, ly = threadIdx.y;
    const int tid = ly * Ls + s, nthr = Ls * SB;
    const long long N = FULL ? 2 * g.Vh : g.Vh;
    const long long per = (N + SB - 1) / SB;
    const long long rhs = blockIdx.x / per, base = (blockIdx.x % per) * SB;
    const int live = (int)(N - base < SB ? N - base : SB);  // sites of this block
    const long long site = base + ly;
    int par = 1;
    long long sr = rhs * g.Vh + site;
    if (FULL) {
        long long q = site;
        const int x = (int)(q % g.X); q /= g.X;
        const int y = (int)(q % g.Y); q /= g.Y;
        const int z = (int)(q % g.Z); q /= g.Z;
        par = (x + y + z + (int)q) & 1;
        sr = rhs * g.Vh + (site >> 1);
    }
    double2* row = tile + (size_t)tid * kLayoutRow;
    // a caller's doubles need not be 16-byte aligned (so `user` must not be a double2*: the compiler may then
    // join the two 8-byte accesses)
    const bool wide = (reinterpret_cast<size_t>(user) & 15) == 0;
    // (slice, site of the block, 16-byte word) of the user side, words fastest
    auto copy_user = [&](auto f) {
        for (int i = tid; i < Ls * live * 12; i += nthr) {
            const int w = i % 12, r = i / 12, l = r % live, t = r / live;
            f(user + (((rhs * Ls + t) * N + base + l) * 12 + w) * 2, tile + ((size_t)l * Ls + t) * kLayoutRow + w);
        }
    };
    if (TO_INTERNAL) {
        copy_user([=](const double* u, double2* t) {
            if (wide) *t = __ldg(reinterpret_cast<const double2*>(u));
            else *t = make_double2(__ldg(u), __ldg(u + 1));
        });
        __syncthreads();
        if (ly >= live) return;
        R v[24];
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const double2 d = row[k];
            v[2 * k] = (R)d.x;
            v[2 * k + 1] = (R)d.y;
        }
        if (par) odd.store(sr, s, v);
        else even.store(sr, s, v);
    } else {
        if (ly < live) {
            R v[24];
            if (par) odd.load(sr, s, v);
            else even.load(sr, s, v);
#pragma unroll
            for (int k = 0; k < 12; ++k) row[k] = make_double2((double)v[2 * k], (double)v[2 * k + 1]);
        }
        __syncthreads();
        copy_user([=](double* u, const double2* t) {
            if (wide) {
                *reinterpret_cast<double2*>(u) = *t;
            } else {
                u[0] = t->x;
                u[1] = t->y;
            }
        });
    }
}

// The user's links U[site][mu][9] to the FP64, FP32 and fixed-point copies, per parity and direction (no fixed-point
// copy: fx is null; fx_exp, unless null too, then marks every link as raw). A block takes kPackSites consecutive
// sites; the two sites of a pair (2k, 2k + 1) differ in parity and have the same index k in their copies, so of each
// parity and direction the block writes one contiguous run. Read and written with consecutive 16-byte accesses,
// turned in shared memory. (A thread that walked its link's 144 bytes in every copy took 202 us on 16^3 x 32, 134
// without the fixed-point copy; now 58 us, 4.7 TB/s.)
constexpr int kPackSites = 32, kPackLinks = 4 * kPackSites;
__global__ void __launch_bounds__(kPackLinks) gauge_pack_kernel(double2* u64, float4* u32, int4* fx, int* fx_exp,
                                                                const double* __restrict__ U, Geom g) {
    __shared__ double2 tile[kPackLinks * 9];
    __shared__ int swapped[kPackSites / 2];  // whether site 2k of the block is odd
    __shared__ int exps[kPackLinks];
    const long long base = (long long)blockIdx.x * kPackSites, left = 2 * g.Vh - base;
    const int sites = left < kPackSites ? (int)left : kPackSites, links = 4 * sites, tid = threadIdx.x;
    const double* src = U + base * 72;
    const bool wide = (reinterpret_cast<size_t>(U) & 15) == 0;  // a caller's doubles need not be 16-byte aligned
    for (int i = tid; i < links * 9; i += kPackLinks)
        tile[i] = wide ? __ldg(reinterpret_cast<const double2*>(src) + i)
                       : make_double2(__ldg(src + 2 * i), __ldg(src + 2 * i + 1));
    if (tid < sites / 2) {
        long long q = base + 2 * tid;
        const int x = (int)(q % g.X); q /= g.X;
        const int y = (int)(q % g.Y); q /= g.Y;
        const int z = (int)(q % g.Z); q /= g.Z;
        swapped[tid] = (x + y + z + (int)q) & 1;
    }
    __syncthreads();
    // link r of the block in the order of the copies, r = (parity 4 + mu) sites / 2 + k: its places in the tile and
    // there
    const int half = sites / 2;
    auto place = [&](int r) {
        const int q = r / half, k = r % half;
        return (2 * k + ((q >> 2) ^ swapped[k])) * 4 + (q & 3);
    };
    auto index = [&](int r) { return (long long)(r / half) * g.Vh + base / 2 + r % half; };
    if (!fx && fx_exp && tid < links) fx_exp[index(tid)] = kFxRaw;
    if (fx && tid < links) {
        double v[18];
        const double2* u = tile + place(tid) * 9;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            v[2 * k] = u[k].x;
            v[2 * k + 1] = u[k].y;
        }
        const int e = fx_link_exponent(v);  // kFxRaw: the link is read from the FP64 copy
        exps[tid] = e;
        fx_exp[index(tid)] = e;
    }
    __syncthreads();
    for (int i = tid; i < links * 9; i += kPackLinks) {
        const int r = i / 9, w = i % 9;
        const double2 d = tile[place(r) * 9 + w];
        const long long at = index(r) * 9 + w;
        u64[at] = d;
        if (fx) {
            int4 o = make_int4(0, 0, 0, 0);
            if (exps[r] != kFxRaw) {
                fx_split(fx_mantissa<8>(d.x, exps[r]), o.y, o.x);
                fx_split(fx_mantissa<8>(d.y, exps[r]), o.w, o.z);
            }
            fx[at] = o;
        }
    }
    for (int i = tid; i < links * 5; i += kPackLinks) {  // 18 floats and two zeros
        const int r = i / 5, w = i % 5;
        const double2* u = tile + place(r) * 9 + 2 * w;
        const double2 a = u[0], b = w < 4 ? u[1] : make_double2(0.0, 0.0);
        u32[index(r) * 5 + w] = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
    }
}

// On a t-slab (slab != 0) the t-neighbours across the two faces are marked
// -1 - f, f the site's index within its t-slice (the index of the same
// (x, y, z) in the neighbouring slab's face), so the hops read them from halos.
__global__ void neighbour_kernel(int* nbr, Geom g, int slab) {
    const long long n = 2 * g.Vh;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int par = (int)(i / g.Vh);
        const long long j = i % g.Vh;
        int c[4];
        cb_coords(g, j, par, c);
        const int L[4] = {g.X, g.Y, g.Z, g.T};
        int* o = nbr + i * 8;
        for (int mu = 0; mu < 4; ++mu) {
            int f[4] = {c[0], c[1], c[2], c[3]}, b[4] = {c[0], c[1], c[2], c[3]};
            f[mu] = c[mu] + 1 == L[mu] ? 0 : c[mu] + 1;
            b[mu] = c[mu] == 0 ? L[mu] - 1 : c[mu] - 1;
            o[mu] = (int)cb_index(g, f[0], f[1], f[2], f[3]);
            o[4 + mu] = (int)cb_index(g, b[0], b[1], b[2], b[3]);
        }
        if (slab) {
            const long long face = (long long)g.X * g.Y * g.Z / 2;
            if (c[3] == g.T - 1) o[3] = -1 - (int)(j % face);
            if (c[3] == 0) o[7] = -1 - (int)(j % face);
        }
    }
}

static dim3 grid_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    if (b > 152LL * 64) b = 152LL * 64;
    if (b < 1) b = 1;
    return dim3((unsigned)b);
}

template <int P, bool FULL, bool TO>
static int layout_t(mdwf_ctx* c, void* even, void* odd, const double* user, int nrhs) {
    const Geom& g = c->g;
    const long long N = FULL ? 2 * g.Vh : g.Vh;
    const int SB = 128 / g.Ls;
    LaunchScope scope(c, KB_LAYOUT * 3 + P, (double)nrhs * N * g.Ls * (192.0 + site_bytes(P)), 0.0);
    layout_kernel<P, FULL, TO><<<dim3((unsigned)((N + SB - 1) / SB * nrhs)), dim3(g.Ls, SB),
                                 sizeof(double2) * kLayoutRow * g.Ls * SB, c->stream>>>(
        make_field<P>(even, g, nrhs), make_field<P>(odd, g, nrhs),
        const_cast<double*>(user), g, nrhs);
    return check_launch();
}

int launch_import_odd(mdwf_ctx* c, void* dst, const double* src, int prec, int nrhs) {
    switch (prec) {
        case MDWF_F64: return layout_t<MDWF_F64, false, true>(c, dst, dst, src, nrhs);
        case MDWF_F32: return layout_t<MDWF_F32, false, true>(c, dst, dst, src, nrhs);
        case MDWF_F16N: return layout_t<MDWF_F16N, false, true>(c, dst, dst, src, nrhs);
    }
    return MDWF_EINVAL;
}

int launch_export_odd(mdwf_ctx* c, double* dst, const void* src, int prec, int nrhs) {
    void* f = const_cast<void*>(src);
    switch (prec) {
        case MDWF_F64: return layout_t<MDWF_F64, false, false>(c, f, f, dst, nrhs);
        case MDWF_F32: return layout_t<MDWF_F32, false, false>(c, f, f, dst, nrhs);
        case MDWF_F16N: return layout_t<MDWF_F16N, false, false>(c, f, f, dst, nrhs);
    }
    return MDWF_EINVAL;
}

int launch_split_full(mdwf_ctx* c, void* dst_even, void* dst_odd, const double* full, int prec, int nrhs) {
    switch (prec) {
        case MDWF_F64: return layout_t<MDWF_F64, true, true>(c, dst_even, dst_odd, full, nrhs);
        case MDWF_F32: return layout_t<MDWF_F32, true, true>(c, dst_even, dst_odd, full, nrhs);
        case MDWF_F16N: return layout_t<MDWF_F16N, true, true>(c, dst_even, dst_odd, full, nrhs);
    }
    return MDWF_EINVAL;
}

int launch_join_full(mdwf_ctx* c, double* full, const void* even, const void* odd, int prec, int nrhs) {
    void* e = const_cast<void*>(even);
    void* o = const_cast<void*>(odd);
    switch (prec) {
        case MDWF_F64: return layout_t<MDWF_F64, true, false>(c, e, o, full, nrhs);
        case MDWF_F32: return layout_t<MDWF_F32, true, false>(c, e, o, full, nrhs);
        case MDWF_F16N: return layout_t<MDWF_F16N, true, false>(c, e, o, full, nrhs);
    }
    return MDWF_EINVAL;
}

int launch_gauge_pack(mdwf_ctx* c, const double* U) {
    const long long n = 2 * c->g.Vh * 4;
    LaunchScope scope(c, KB_LAYOUT * 3 + MDWF_F64, n * (144.0 * (c->gauge_fx ? 3 : 2) + 80.0), 0.0);
    gauge_pack_kernel<<<(unsigned)((2 * c->g.Vh + kPackSites - 1) / kPackSites), kPackLinks, 0, c->stream>>>(
        (double2*)c->gauge[0], (float4*)c->gauge[1], (int4*)c->gauge_fx, c->gauge_fx_exp, U, c->g);
    return check_launch();
}

}  // namespace mdwf

namespace mdwf {
int launch_build_neighbours(mdwf_ctx* c) {
    const long long n = 2 * c->g.Vh;
    LaunchScope scope(c, KB_LAYOUT * 3 + MDWF_F64, n * 32.0, 0.0);
    neighbour_kernel<<<grid_for(n, 256), 256, 0, c->stream>>>(c->nbr, c->g, c->slab ? 1 : 0);
    return check_launch();
}
}  // namespace mdwf
