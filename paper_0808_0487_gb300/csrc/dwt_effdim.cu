// dwt_effdim.cu -- the class partials of every tile -> variances and effective
// dimensions (Sec. 4), one launch for a batch.
#include <cooperative_groups.h>

#include <algorithm>

#include "dwt_effdim.cuh"

namespace dwt {

// One cluster of CL CTAs per function (CL = 1: an ordinary CTA).  A warp sums
// whole classes: lane l takes the tiles l, l + 32, ... (eight loads in flight),
// then a fixed tree, all in FP64, so the result depends on nothing but the
// partials.  The totals meet in the first CTA's shared memory, which forms the
// outputs.  It replaces a launch of one CTA per class and function followed by
// one of one warp per function: small nets are bound by the second launch and
// by that warp's serial loop (p = 2, m = 17, s = 24, 7 functions: 14.5 us for
// the two), large ones by the reads of the partials (1 MB per function at
// m = 24, s = 32).
constexpr int kRedThreads = 512;

template <int CL>
__global__ void __launch_bounds__(kRedThreads) k_effdim_reduce(const double* __restrict__ part, long long nchunk,
                                                               int nb, double thr, EffOut o, long long f0) {
    namespace cg = cooperative_groups;
    __shared__ double c[2 * 256];
    __shared__ int first[2];
    const int nb2 = 2 * nb, lane = threadIdx.x & 31;
    const long long fn = f0 + blockIdx.y;
    double* dst = c;
    if constexpr (CL > 1) {
        dst = cg::this_cluster().map_shared_rank(c, 0);
        cg::this_cluster().sync();   // the first CTA is running before its shared memory is written
    }
    for (int b = blockIdx.x * (kRedThreads / 32) + (threadIdx.x >> 5); b < nb2; b += CL * (kRedThreads / 32)) {
        const double* p = part + (fn * nb2 + b) * nchunk;
        double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        long long t = lane;
        for (; t + 7 * 32 < nchunk; t += 8 * 32) {
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] += p[t + 32 * i];
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (t + 32 * i < nchunk) acc[i] += p[t + 32 * i];
        double x = ((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7]));
#pragma unroll
        for (int h = 16; h > 0; h >>= 1) x += __shfl_xor_sync(0xffffffffu, x, h);
        if (lane == 0) dst[b] = x;
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
        DWT_CK(cudaLaunchKernelEx(&cfg, k_effdim_reduce<CL>, part, nchunk, nb, thr, o, (long long)f0));
    }
    DWT_CK_LAUNCH("k_effdim_reduce");
    return DWT_OK;
}

int effdim_reduce(const double* part, long long nchunk, int nb, int batch, double thr, const EffOut& o,
                  cudaStream_t st) {
    if (!o.vt && !o.vs && !o.dt && !o.ds) return DWT_OK;
    // one CTA reads about 100 GB/s of partials: past 128 KB per function a
    // cluster of eight shares them
    if (2ll * nb * nchunk <= 16384) return launch_reduce<1>(part, nchunk, nb, batch, thr, o, st);
    return launch_reduce<8>(part, nchunk, nb, batch, thr, o, st);
}

}  // namespace dwt
