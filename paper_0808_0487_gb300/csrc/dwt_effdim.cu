// dwt_effdim.cu -- the class partials of every tile -> variances and effective
// dimensions (Sec. 4), one launch for a batch.
#include <cooperative_groups.h>

#include <algorithm>

#include "dwt_effdim.cuh"

namespace dwt {

// One cluster of CL CTAs per function (CL = 1: an ordinary CTA).  The class
// totals meet in the first CTA's shared memory, which forms the outputs.
// p = 2, m = 17, s = 24, 7 functions: 4.3 us, m = 20, s = 16, 32 functions:
// 4.9 us in a graph, where the two launches that this one replaces took about
// 11 us.
constexpr int kRedThreads = 512;

template <int CL>
__global__ void __launch_bounds__(kRedThreads) k_effdim_reduce(const double* __restrict__ part, long long nchunk,
                                                               int nb, int lg, double thr, EffOut o, long long f0) {
    namespace cg = cooperative_groups;
    chain_begin();
    __shared__ double c[2 * 256];
    __shared__ int first[2];
    const int nb2 = 2 * nb;
    const long long fn = f0 + blockIdx.y;
    double* dst = c;
    if constexpr (CL > 1) {
        dst = cg::this_cluster().map_shared_rank(c, 0);
        cg::this_cluster().sync();   // the first CTA is running before its shared memory is written
    }
    sum_rows(part + fn * nb2 * nchunk, nb2, (int)nchunk, lg, blockIdx.x, CL, dst);
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
    const int lg = sum_rows_lanes((2 * nb + CL - 1) / CL, nchunk, kRedThreads);
    for (int f0 = 0; f0 < batch; f0 += 65535) {
        LaunchScope ls("effdim_reduce", st);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(CL, (unsigned)std::min(65535, batch - f0));
        cfg.blockDim = dim3(kRedThreads);
        cfg.stream = st;
        cudaLaunchAttribute at[2];   // as launch_chain, in clusters
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        at[1].id = cudaLaunchAttributeClusterDimension;
        at[1].val.clusterDim = {CL, 1, 1};
        cfg.attrs = at;
        cfg.numAttrs = CL > 1 ? 2 : 1;
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
