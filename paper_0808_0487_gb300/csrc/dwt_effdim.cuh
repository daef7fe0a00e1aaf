// dwt_effdim.cuh -- class totals -> cumulative variances and effective
// dimensions (Sec. 4), shared by the reduction of tile partials and by kernels
// that hold a function's class totals in shared memory.  Internal to libdwt.
#pragma once

#include "dwt_internal.cuh"

namespace dwt {

// Sums of the rows rank, rank + nranks, ... of part [rows][n] into dst[row], by
// all threads of a CTA.  2^lg lanes share a row: lane l adds the entries l,
// l + 2^lg, ... in order, a fixed tree adds the lanes, all in FP64, so the
// result depends on nothing but the entries.  The FP64 pipe bounds it (an SM
// starts a warp's addition every 19 cycles, and one takes 64): a row takes as
// many lanes as the CTA has to spare and no more, since a lane without an entry
// costs as much as one with (50 rows of 16: a warp per row 12 us, two lanes 4.3).
__device__ __forceinline__ void sum_rows(const double* part, int rows, int n, int lg, int rank, int nranks,
                                         double* dst) {
    const int t = threadIdx.x, lane = t & ((1 << lg) - 1), step = 1 << lg;
    // whole warps go round together (the tree's shuffles need all their lanes)
    for (int b0 = ((t & ~31) >> lg) * nranks; b0 < rows; b0 += ((int)blockDim.x >> lg) * nranks) {
        const int b = b0 + ((t & 31) >> lg) * nranks + rank;
        double x = 0.0;
        if (b < rows) {
            const double* p = part + (long long)b * n;
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
        for (int h = step >> 1; h > 0; h >>= 1) x += __shfl_xor_sync(0xffffffffu, x, h);
        if (lane == 0 && b < rows) dst[b] = x;
    }
}

// lg for `rows` rows of n entries in a CTA of `threads`: eight entries per lane at least
static inline int sum_rows_lanes(int rows, long long n, int threads) {
    int lg = 0;
    while (lg < 5 && rows << (lg + 1) <= threads && (16ll << lg) <= n) ++lg;
    return lg;
}

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
