// dwt_effdim.cu -- the class partials of every tile -> variances and effective
// dimensions (Sec. 4), one launch for a batch.
#include <cooperative_groups.h>

#include <algorithm>

#include "dwt_effdim.cuh"

namespace dwt {

// One cluster of CL CTAs per function (CL = 1: an ordinary CTA).  2^lg lanes
// share a class: lane l adds the tiles l, l + 2^lg, ... in order, a fixed tree
// adds the lanes, all in FP64, so the result depends on nothing but the
// partials.  The totals meet in the first CTA's shared memory, which forms the
// outputs.  The FP64 pipe bounds it (an SM starts a warp's addition about every
// 16 cycles): a class takes as many lanes as the CTA has to spare and no more,
// since a lane without a tile costs as much as one with (p = 2, m = 17, s = 24,
// 7 functions: a warp per class 12 us, this form 4.3 us; m = 20, s = 16, 32
// functions: 4.9 us; in a graph, where the two launches that this one replaces
// took about 11 us).
constexpr int kRedThreads = 512;

template <int CL>
__global__ void __launch_bounds__(kRedThreads) k_effdim_reduce(const double* __restrict__ part, long long nchunk,
                                                               int nb, int lg, double thr, EffOut o, long long f0) {
    namespace cg = cooperative_groups;
    __shared__ double c[2 * 256];
    __shared__ int first[2];
    const int nb2 = 2 * nb;
    const long long fn = f0 + blockIdx.y;
    double* dst = c;
    if constexpr (CL > 1) {
        dst = cg::this_cluster().map_shared_rank(c, 0);
        cg::this_cluster().sync();   // the first CTA is running before its shared memory is written
    }
    // this CTA's classes: blockIdx.x, + CL, ...; whole warps go round together
    // (the tree's shuffles need all their lanes)
    const int t = threadIdx.x, lane = t & ((1 << lg) - 1);
    for (int b0 = ((t & ~31) >> lg) * CL; b0 < nb2; b0 += (kRedThreads >> lg) * CL) {
        const int b = b0 + ((t & 31) >> lg) * CL + blockIdx.x;
        double x = 0.0;
        if (b < nb2) {
            const double* p = part + (fn * nb2 + b) * nchunk;
            const int n = (int)nchunk, step = 1 << lg;
            int i = lane;
            for (; i + 7 * step < n; i += 8 * step) {   // eight loads in flight
                double r[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) r[k] = p[i + k * step];
#pragma unroll
                for (int k = 0; k < 8; ++k) x += r[k];
            }
            double r[7];
#pragma unroll
            for (int k = 0; k < 7; ++k) r[k] = i + k * step < n ? p[i + k * step] : 0.0;
#pragma unroll
            for (int k = 0; k < 7; ++k)
                if (i + k * step < n) x += r[k];
        }
        for (int h = (1 << lg) >> 1; h > 0; h >>= 1) x += __shfl_xor_sync(0xffffffffu, x, h);
        if (lane == 0 && b < nb2) dst[b] = x;
    }
    if constexpr (CL > 1) {
        cg::this_cluster().sync();
        if (blockIdx.x != 0) return;
    } else {
        __syncthreads();
    }
    effdim_outputs(c, first, nb, thr, o, fn);
}

template <int CL>
static int launch_reduce(const double* part, long long nchunk, int nb, int batch, double thr, const EffOut& o,
                         cudaStream_t st) {
    const int per = (2 * nb + CL - 1) / CL;
    int lg = 0;   // lanes of a class: within a CTA's threads, eight tiles per lane at least
    while (lg < 5 && per << (lg + 1) <= kRedThreads && (16ll << lg) <= nchunk) ++lg;
    for (int f0 = 0; f0 < batch; f0 += 65535) {
        LaunchScope ls("effdim_reduce", st);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(CL, (unsigned)std::min(65535, batch - f0));
        cfg.blockDim = dim3(kRedThreads);
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim = {CL, 1, 1};
        cfg.attrs = at;
        cfg.numAttrs = CL > 1 ? 1 : 0;
        DWT_CK(cudaLaunchKernelEx(&cfg, k_effdim_reduce<CL>, part, nchunk, nb, lg, thr, o, (long long)f0));
    }
    DWT_CK_LAUNCH("k_effdim_reduce");
    return DWT_OK;
}

int effdim_reduce(const double* part, long long nchunk, int nb, int batch, double thr, const EffOut& o,
                  cudaStream_t st) {
    if (!o.vt && !o.vs && !o.dt && !o.ds) return DWT_OK;
    // an SM adds about 3 partials a nanosecond; a cluster costs about 0.8 us to
    // start and join: 800 partials 4.3 us in one CTA, 5.0 in a cluster, 7398 5.7
    // and 4.4
    if (2ll * nb * nchunk <= 2048) return launch_reduce<1>(part, nchunk, nb, batch, thr, o, st);
    return launch_reduce<8>(part, nchunk, nb, batch, thr, o, st);
}

}  // namespace dwt
