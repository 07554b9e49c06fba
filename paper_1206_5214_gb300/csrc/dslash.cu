// Hop launch dispatch over the operator precisions (the kernels are in
// hop_kernel.cuh, instantiated in dslash_f64.cu, dslash_f32.cu and
// dslash_f16n.cu), the block shapes of the hop kernels, and the self-test of
// the bounded device-side wait.
#include "mdwf_internal.cuh"
#include "mbarrier.cuh"

namespace mdwf {

template <int P> int launch_hop_t(mdwf_ctx* c, const HopLaunch& h);

// The block shape of a hop launch: as many whole s-columns as fit 128 threads, or the autotuned number. Where such
// blocks are so few that the time of a hop is that of one thread's chain of eight neighbours, four or (FP64) two
// threads share a column (STAGE 5 and 6 of the kernel) and a block holds a fourth or half of the columns. M alone in
// us, one, two and four threads a column, by the number of ordinary blocks on 152 SMs:
//   FP32: 8 blocks 16.4, -, 13.7; 128 blocks 17.0, -, 14.4; 140 blocks 20.5, -, 16.5; 256 blocks 16.5, -, 20.5
//   FP64: 8 blocks 47, 34, 30; 64 blocks 49, 34, 34; 128 blocks 49, 43, 56; 205 blocks 64, 46, 72;
//         256 blocks 64, 77, 95
// FP32 gains while the ordinary form leaves an SM at most one block. The FP64 split forms run three blocks per SM:
// two threads a column pay while those blocks are one wave (205 blocks make 410, 256 make 512, of 456), four while
// the integer pipe is not the limit.
// Not for FP16+norm (its sums would round differently) or a chosen load strategy. A tuned number of sites that is the
// split form's selects that form (so the tuner, whose candidates hold it, can choose it); any other the ordinary one.
HopShape hop_shape(const mdwf_ctx* c, int prec, int nrhs) {
    const int full = 128 / c->g.Ls, tuned = nrhs >= 1 && nrhs <= 64 ? c->sb_tune[prec][nrhs] : 0;
    const long long blocks = (c->g.Vh + full - 1) / full * nrhs;
    int split = 1;
    if (prec == MDWF_F32 && blocks <= c->sms) split = 4;
    if (prec == MDWF_F64) split = blocks * 152 <= c->sms * 64 ? 4 : blocks * 2 <= c->sms * 3 ? 2 : 1;
    if (c->slab || c->hop_stage[prec] != 0) split = 1;
    const int sites = 128 / split / c->g.Ls;
    return tuned > 0 && tuned != sites ? HopShape{tuned, 1} : HopShape{sites, split};
}

// The fused iteration drops its t field when the FUSE_R epilogue can rebuild
// t = I^dag v by shuffles: FP32 or FP16+norm operators at Ls = 16 with the
// closed-form s-operators, whole s-columns in every warp (an even number of
// sites per block) and a load strategy whose kernels fix Ls = 16 at compile
// time (not the two shared-memory staging modes).
bool hop_no_t_ok(const mdwf_ctx* c, int prec, int nrhs) {
    if (prec == MDWF_F64 || c->g.Ls != 16 || c->dense_s || c->sdep) return false;
    if (hop_shape(c, prec, nrhs).sites & 1) return false;
    const int mode = c->hop_stage[prec];
    return mode != 1 && mode != 2;
}

int hop_blocks(const mdwf_ctx* c, int prec, int nrhs) {
    const int SB = hop_shape(c, prec, nrhs).sites;
    return (int)((c->g.Vh + SB - 1) / SB);
}

// One thread waits, bounded, on an mbarrier that expects two arrivals of
// which `arrivals` are made; a wait that gives up sets the error word.
__global__ void k_wait_selftest(int* err, int arrivals) {
    __shared__ unsigned long long bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 2);
    mbar_init_fence();
    for (int k = 0; k < arrivals; ++k) mbar_arrive(&bar);
    if (!mbar_wait(&bar, 0)) atomicOr(err, 1);
}

int launch_hop(mdwf_ctx* c, int prec, const HopLaunch& h) {
    switch (prec) {
        case MDWF_F64: return launch_hop_t<MDWF_F64>(c, h);
        case MDWF_F32: return launch_hop_t<MDWF_F32>(c, h);
        case MDWF_F16N: return launch_hop_t<MDWF_F16N>(c, h);
    }
    return MDWF_EINVAL;
}

}  // namespace mdwf

using namespace mdwf;

extern "C" int mdwf_selftest_wait(mdwf_ctx* c, int arrivals) {
    if (!c || arrivals < 0 || arrivals > 2) return MDWF_EINVAL;
    int st;
    if ((st = cuda_status(cudaSetDevice(c->device)))) return st;
    k_wait_selftest<<<1, 32, 0, c->stream>>>(c->dev_err, arrivals);
    if ((st = check_launch())) return st;
    return device_wait_status(c);
}
