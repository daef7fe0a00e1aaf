// dwt_effdim.cuh -- class totals -> cumulative variances and effective
// dimensions (Sec. 4), shared by the reduction of tile partials and by kernels
// that hold a function's class totals in shared memory.  Internal to libdwt.
#pragma once

#include "dwt_internal.cuh"

namespace dwt {

// c: the 2 nb class totals of function fn in shared memory (truncation
// classes, then support sizes), complete and visible to the block; first: two
// ints of shared memory.  All threads of the block call it.  The cumulative
// sums are formed in class order (one lane each), so that classes that add
// nothing leave them unchanged; the comparisons and stores run in parallel.
// The chain of nb dependent FP64 additions bounds it (about 1 us at nb = 33).
__device__ __forceinline__ void effdim_outputs(double* c, int* first, int nb, double thr, const EffOut& o,
                                               long long fn) {
    const int t = threadIdx.x;
    if (t < 2) {
        first[t] = nb;
        double* x = c + t * nb;
        double acc = 0.0;
        for (int d0 = 0; d0 < nb; d0 += 8) {
            double r[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) r[i] = d0 + i < nb ? x[d0 + i] : 0.0;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (d0 + i < nb) x[d0 + i] = acc += r[i];
        }
    }
    __syncthreads();
    for (int i = t; i < 2 * nb; i += blockDim.x) {
        const int k = i >= nb, d = i - k * nb;
        const double tot = c[nb - 1];
        if (!k && o.vt) o.vt[fn * o.vstride + d] = c[i];
        if (k && o.vs) o.vs[fn * o.vstride + d] = c[i];
        if (tot > 0.0 && c[i] >= thr * tot) atomicMin(first + k, d);
    }
    __syncthreads();
    if (t == 0) {
        if (o.dt) o.dt[fn * o.dstride] = first[0] < nb ? first[0] : 0;
        if (o.ds) o.ds[fn * o.dstride] = first[1] < nb ? first[1] : 0;
    }
}

}  // namespace dwt
