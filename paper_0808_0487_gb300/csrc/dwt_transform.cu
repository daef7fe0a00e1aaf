// dwt_transform.cu -- the transforms and the interpolation: which kernels run
// a call (register tiles, FP64 integer stages or one-launch form for p = 2, the
// generic passes of dwt_pass.cuh otherwise), and the effective dimension of
// given coefficients (Sec. 4).
#include "dwt_pass.cuh"

namespace dwt {

bool p2_fast_ok(int m);
bool p2_interp_ok(int m, int s);
int p2_transform(dwt_plan_s* Pl, const void* in, void* out, int batch, long long ld_in, long long ld_out,
                 dwt_dtype t, int sgn, cudaStream_t st);
int p2_interpolate(dwt_plan_s* Pl, const float* f, float* c, float* coef, int batch, long long ld, const float* W,
                   bool tc, double** part_out, long long* ntile_out, cudaStream_t st);

bool p2d_ok(int m);
int p2d_transform(dwt_plan_s* Pl, const double* in, double* out, int batch, long long ld_in, long long ld_out,
                  int sgn, cudaStream_t st);
int p2d_grouped(const std::vector<GroupJob>& jobs, int sgn, cudaStream_t st);
bool p2_small_ok(int m);
int p2_small_interpolate(dwt_plan_s* Pl, const float* f, float* c, float* coef, int batch, long long ld,
                         bool weighted, double thr, const EffOut& o, cudaStream_t st);

static bool aligned16(const void* p, long long ld, int elem) {
    return ((uintptr_t)p & 15) == 0 && ((ld * elem) & 15) == 0;
}
// the passes of each prime (dwt_pass_p<P>.cu)
#define DWT_EACH_PRIME(X) X(2) X(3) X(5) X(7) X(11) X(13) X(17) X(19) X(23) X(29) X(31)
#define DWT_EXTERN(P)                                                                                             \
    extern template int transform_p<P>(dwt_plan_s*, const void*, void*, int, long long, long long, dwt_dtype,     \
                                       dwt_dtype, int, cudaStream_t);                                             \
    extern template int digits_p<P>(dwt_plan_s*, const void*, void*, int, long long, long long, dwt_dtype,        \
                                    dwt_dtype, int, int, int, cudaStream_t);                                      \
    extern template int grouped_p<P>(const std::vector<GroupJob>&, dwt_dtype, dwt_dtype, int, cudaStream_t);      \
    extern template int interpolate_p<P>(dwt_plan_s*, const void*, void*, void*, int, long long, dwt_dtype,       \
                                         dwt_weight, double*, int*, double, cudaStream_t);
DWT_EACH_PRIME(DWT_EXTERN)

// class sums of given coefficients: grid (chunks, functions), 8192 elements per chunk
template <typename T>
__global__ void __launch_bounds__(256) k_effdim_bins(const T* coef, long long ld, long long N, const uint8_t* cls,
                                                     int nb, long long nchunk, double* part) {
    extern __shared__ __align__(16) unsigned char smraw[];
    float* bins = reinterpret_cast<float*>(smraw);
    const int nb2 = 2 * nb, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    chain_begin();
    for (int i = threadIdx.x; i < (int)(blockDim.x >> 5) * nb2 * 32; i += blockDim.x) bins[i] = 0.f;
    __syncthreads();
    const long long fn = blockIdx.y, chunk = blockIdx.x;
    const long long h0 = chunk * 8192, h1 = min(N, h0 + 8192);
    float* mybins = bins + (size_t)w * nb2 * 32 + lane;
    const T* g = coef + fn * ld;
    for (long long H = h0 + threadIdx.x; H < h1; H += blockDim.x) {
        if (H == 0) continue;
        const float q = mag2<T>(g[H]);
        const uchar2 k = __ldg(reinterpret_cast<const uchar2*>(cls) + H);
        mybins[(int)k.x * 32] += q;
        mybins[(nb + (int)k.y) * 32] += q;
    }
    __syncthreads();
    reduce_bins(bins, nb2, blockDim.x >> 5, part + fn * nb2 * nchunk + chunk, nchunk);
}
int run_transform_digits(dwt_plan_s* Pl, const void* in, void* out, int batch, long long ld_in, long long ld_out,
                         dwt_dtype in_t, dwt_dtype out_t, int d0, int nd, int sgn, cudaStream_t st) {
#define DWT_CASE(P) case P: return digits_p<P>(Pl, in, out, batch, ld_in, ld_out, in_t, out_t, d0, nd, sgn, st);
    switch (Pl->p) {
        DWT_EACH_PRIME(DWT_CASE)
        default: set_error("unsupported p"); return DWT_EUNSUPPORTED;
    }
#undef DWT_CASE
}
// Grouped transforms of jobs that share p and the element types (checked by
// the caller).  p = 2 jobs that their own call sends to the register-tile
// kernels go there too: m = 12 .. 14 as one grouped low pass per tile size,
// larger ones one call each; FP64 ones of 2^12 points and more run their integer
// passes grouped; all other jobs run the generic passes grouped.
int run_transform_grouped(const std::vector<GroupJob>& jobs, dwt_dtype in_t, dwt_dtype out_t, int sgn,
                          cudaStream_t st) {
    if (jobs.empty()) return DWT_OK;
    const int p = jobs[0].plan->p;
    std::vector<GroupJob> generic, wide, lo[3];
    for (const GroupJob& j : jobs) {
        if (j.batch <= 0) continue;
        if (p == 2 && (in_t == DWT_F32 || in_t == DWT_I32) && p2_fast_ok(j.plan->m) && aligned16(j.in, j.ld_in, 4) &&
            aligned16(j.out, j.ld_out, 4)) {
            if (j.plan->m <= 14) {
                lo[j.plan->m - 12].push_back(j);
            } else {
                const int rc = p2_transform(j.plan, j.in, j.out, j.batch, j.ld_in, j.ld_out, in_t, sgn, st);
                if (rc) return rc;
            }
            continue;
        }
        if (p == 2 && in_t == DWT_F64 && p2d_ok(j.plan->m)) {
            wide.push_back(j);
            continue;
        }
        generic.push_back(j);
    }
    for (int L = 12; L <= 14; ++L)
        if (!lo[L - 12].empty()) {
            const int rc = p2_lo_grouped(L, lo[L - 12], in_t, sgn, st);
            if (rc) return rc;
        }
    if (!wide.empty()) {
        const int rc = p2d_grouped(wide, sgn, st);
        if (rc) return rc;
    }
    if (generic.empty()) return DWT_OK;
#define DWT_CASE(P) case P: return grouped_p<P>(generic, in_t, out_t, sgn, st);
    switch (p) {
        DWT_EACH_PRIME(DWT_CASE)
        default: set_error("unsupported p"); return DWT_EUNSUPPORTED;
    }
#undef DWT_CASE
}

int run_transform(dwt_plan_s* Pl, const void* in, void* out, int batch, long long ld_in, long long ld_out,
                  dwt_dtype in_t, dwt_dtype out_t, int sgn, cudaStream_t st) {
    if (Pl->p == 2 && (in_t == DWT_F32 || in_t == DWT_I32) && p2_fast_ok(Pl->m) && aligned16(in, ld_in, 4) &&
        aligned16(out, ld_out, 4))
        return p2_transform(Pl, in, out, batch, ld_in, ld_out, in_t, sgn, st);
    if (Pl->p == 2 && in_t == DWT_F64 && p2d_ok(Pl->m))
        return p2d_transform(Pl, (const double*)in, (double*)out, batch, ld_in, ld_out, sgn, st);
#define DWT_CASE(P) case P: return transform_p<P>(Pl, in, out, batch, ld_in, ld_out, in_t, out_t, sgn, st);
    switch (Pl->p) {
        DWT_EACH_PRIME(DWT_CASE)
        default: set_error("unsupported p"); return DWT_EUNSUPPORTED;
    }
#undef DWT_CASE
}
int run_interpolate(dwt_plan_s* Pl, const void* f, void* c, void* coef, int batch, long long ld, dwt_dtype f_t,
                    dwt_weight weight, dwt_algo algo, double* var, int* dim, double thr, cudaStream_t st) {
    const bool fast = Pl->p == 2 && p2_interp_ok(Pl->m, Pl->s) && aligned16(f, ld, 4) && aligned16(c, ld, 4);
    if (algo == DWT_ALGO_TC_SPLIT_BF16 && !(fast && Pl->m >= 18)) {
        set_error("the tensor-core interpolation needs p = 2, 18 <= m <= 24 and 16-byte aligned rows");
        return DWT_EUNSUPPORTED;
    }
    if (fast && Pl->d_tkt) {
        double* part = nullptr;
        long long ntile = 0;
        int rc = p2i_interpolate(Pl, (const float*)f, (float*)c, (float*)coef, batch, ld,
                                 weight == DWT_WEIGHT_INV_SQ_WAVENUMBER, algo == DWT_ALGO_TC_SPLIT_BF16, &part, &ntile,
                                 st);
        if (rc) return rc;
        return effdim_reduce(part, ntile, Pl->s + 1, batch, thr, eff_packed(var, dim, Pl->s + 1), st);
    }
    if (fast) {
        double* part = nullptr;
        long long ntile = 0;
        int rc = p2_interpolate(Pl, (const float*)f, (float*)c, (float*)coef, batch, ld,
                                weight == DWT_WEIGHT_INV_SQ_WAVENUMBER ? Pl->d_W : nullptr,
                                algo == DWT_ALGO_TC_SPLIT_BF16, &part, &ntile, st);
        if (rc) return rc;
        return effdim_reduce(part, ntile, Pl->s + 1, batch, thr, eff_packed(var, dim, Pl->s + 1), st);
    }
    if (Pl->p == 2 && p2_small_ok(Pl->m))
        return p2_small_interpolate(Pl, (const float*)f, (float*)c, (float*)coef, batch, ld,
                                    weight == DWT_WEIGHT_INV_SQ_WAVENUMBER, thr, eff_packed(var, dim, Pl->s + 1), st);
#define DWT_CASE(P) case P: return interpolate_p<P>(Pl, f, c, coef, batch, ld, f_t, weight, var, dim, thr, st);
    switch (Pl->p) {
        DWT_EACH_PRIME(DWT_CASE)
        default: set_error("unsupported p"); return DWT_EUNSUPPORTED;
    }
#undef DWT_CASE
}

template <typename T>
static int effdim_t(dwt_plan_s* Pl, const void* coef, int batch, long long ld, const EffOut& o, double thr,
                    cudaStream_t st) {
    const int nb = Pl->s + 1, nb2 = 2 * nb;
    const long long nchunk = (Pl->N + 8191) / 8192;
    const int nw = bins_warps(0, nb2);
    if (nw < 1) {
        set_error("s = %d too large for the variance pass", Pl->s);
        return DWT_EUNSUPPORTED;
    }
    const size_t smem = (size_t)nw * nb2 * 32 * 4;
    int rc = ensure_workspace(Pl, (size_t)batch * nchunk * nb2 * sizeof(double), st);
    if (rc) return rc;
    double* part = (double*)Pl->d_ws;
    auto kern = k_effdim_bins<T>;
    rc = set_smem(kern, smem);
    if (rc) return rc;
    for (int f0 = 0; f0 < batch; f0 += 65535) {
        const int nf = std::min(65535, batch - f0);
        LaunchScope ls("effdim_bins", st);
        launch_chain(kern, dim3((unsigned)nchunk, (unsigned)nf), nw * 32, smem, st,
            (const T*)coef + (long long)f0 * ld, ld, Pl->N, Pl->d_cls, nb, nchunk, part + (long long)f0 * nchunk * nb2);
    }
    DWT_CK_LAUNCH("k_effdim_bins");
    return effdim_reduce(part, nchunk, nb, batch, thr, o, st);
}

// The class sums of effdim_t, with the partials and totals in a scratch array
// supplied by the caller (cap doubles) instead of the plan's workspace:
// functions go through in groups whose partials fit, one group after another
// on the stream, so the array is reused in stream order.  Makes no allocation.
template <typename T>
static int effdim_scratch_t(dwt_plan_s* Pl, const void* coef, int batch, long long ld, double* var, int* dim,
                            double thr, double* scratch, long long cap, cudaStream_t st) {
    const int nb = Pl->s + 1, nb2 = 2 * nb;
    const long long nchunk = (Pl->N + 8191) / 8192;
    const long long per = (long long)nb2 * (nchunk + 1);
    const int nw = bins_warps(0, nb2);
    if (nw < 1 || per > cap) {
        set_error("class partials of one function do not fit the scratch array");
        return DWT_EINVAL;
    }
    const size_t smem = (size_t)nw * nb2 * 32 * 4;
    auto kern = k_effdim_bins<T>;
    int rc = set_smem(kern, smem);
    if (rc) return rc;
    const int G = (int)std::min<long long>(std::min<long long>(cap / per, 65535), batch);
    for (int f0 = 0; f0 < batch; f0 += G) {
        const int nf = std::min(G, batch - f0);
        {
            LaunchScope ls("effdim_bins", st);
            launch_chain(kern, dim3((unsigned)nchunk, (unsigned)nf), nw * 32, smem, st,
            (const T*)coef + (long long)f0 * ld, ld, Pl->N, Pl->d_cls, nb, nchunk, scratch);
        }
        DWT_CK_LAUNCH("k_effdim_bins");
        rc = effdim_reduce(scratch, nchunk, nb, nf, thr, eff_packed(var ? var + (long long)f0 * 2 * nb : nullptr,
                                                                dim ? dim + (long long)f0 * 2 : nullptr, nb),
                      st);
        if (rc) return rc;
    }
    return DWT_OK;
}

int effdim_into_scratch(dwt_plan_s* Pl, const void* coef, int batch, long long ld, dwt_dtype t, double* var, int* dim,
                        double thr, double* scratch, long long cap, cudaStream_t st) {
    if (t == DWT_F32) return effdim_scratch_t<float>(Pl, coef, batch, ld, var, dim, thr, scratch, cap, st);
    return effdim_scratch_t<float2>(Pl, coef, batch, ld, var, dim, thr, scratch, cap, st);
}

int run_effdim(dwt_plan_s* Pl, const void* coef, int batch, long long ld, dwt_dtype t, const EffOut& o, double thr,
               cudaStream_t st) {
    if (t == DWT_F32) return effdim_t<float>(Pl, coef, batch, ld, o, thr, st);
    return effdim_t<float2>(Pl, coef, batch, ld, o, thr, st);
}

}  // namespace dwt
