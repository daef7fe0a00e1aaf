// dwt_p2s.cu -- the p = 2 interpolation step of small nets, 2^8 .. 2^14
// points, in one launch: one CTA per function holds the function from its
// samples to its results (forward stages, scale, weight, class sums, inverse
// stages, variances and effective dimensions; Algorithms 1 and 2, Sec. 4).
//
// A small net is bound by latency: the bytes of 2^12 points move in 5 ns, the
// launches and the chain of stages take microseconds.  So the stages run in
// phases of K digits, 2^K elements per thread in registers, with as many
// threads as that leaves (K = 4: 256 threads at 2^12 points), one exchange
// through shared memory between phases; the weights and classes are requested
// before the first stage; the inverse starts on the registers that the forward
// ended with; and the class totals, being those of the only tile, become the
// outputs in the same launch.
//
// Digits are taken in the order of the generic pass it takes the place of (the
// five top ones, then from the lowest), and the class sums keep that pass's
// lanes (nwb warps; lane l of warp w adds the elements w 32 + l, + 32 nwb, ...
// in order; warps in order, then a tree over the lanes), so coefficients and
// variances are the same to the last bit.
#include <algorithm>

#include "dwt_effdim.cuh"

namespace dwt {

namespace {

struct SmallArgs {
    const float* f;
    float* c;
    float* coef;             // optional weighted coefficients
    const float* W;          // NULL: weight 1
    const uint8_t* cls;      // [N][2]
    long long ld;
    float scale;             // 2^-m
    int nb, nwb;             // classes; warps that bin (0: no variances asked for)
    double thr;
    EffOut o;
};

// digits of the phases: position i of the order is digit m - 5 + i (i < 5), then i - 5
template <int M> struct Small {
    static constexpr int K = M == 8 ? 3 : M <= 12 ? 4 : 5;
    static constexpr int NT = 1 << (M - K);
    static constexpr int NPH = (M + K - 1) / K;
    static constexpr int order(int i) { return i < 5 ? M - 5 + i : i - 5; }
    static constexpr int staged(int ph) { return M - ph * K < K ? M - ph * K : K; }
    // digit of register bit i in phase ph: the staged ones in order, then the
    // highest of the others (so that neighbouring threads keep the low digits)
    static constexpr int digit(int ph, int i) {
        if (i < staged(ph)) return order(ph * K + i);
        int left = i - staged(ph);
        for (int d = M - 1; d >= 0; --d) {
            bool used = false;
            for (int k = 0; k < staged(ph); ++k) used = used || order(ph * K + k) == d;
            if (used) continue;
            if (left == 0) return d;
            --left;
        }
        return 0;
    }
    static constexpr unsigned mask(int ph) {
        unsigned v = 0;
        for (int i = 0; i < K; ++i) v |= 1u << digit(ph, i);
        return v;
    }
    // element offset of register r
    static constexpr int off(int ph, int r) {
        int e = 0;
        for (int i = 0; i < K; ++i)
            if ((r >> i) & 1) e |= 1 << digit(ph, i);
        return e;
    }
};

// shared-memory position: e and off have no bits in common, so positions add up
__host__ __device__ constexpr int spos(int e) { return e + (e >> 5); }

// bits of t spread over the digits that phase PH leaves to the threads
template <int M, int PH> __device__ __forceinline__ int thread_base(int t) {
    constexpr unsigned mask = Small<M>::mask(PH);
    int e = 0, k = 0;
#pragma unroll
    for (int d = 0; d < M; ++d)
        if (!((mask >> d) & 1)) {
            e |= ((t >> k) & 1) << d;
            ++k;
        }
    return e;
}

template <int M, int PH, int I = 0> __device__ __forceinline__ void stages(float* v) {
    using G = Small<M>;
    if constexpr (I < G::staged(PH)) {
#pragma unroll
        for (int r = 0; r < (1 << G::K); ++r) {
            if (r & (1 << I)) continue;
            const float a = v[r], b = v[r | (1 << I)];
            v[r] = a + b;
            v[r | (1 << I)] = a - b;
        }
        stages<M, PH, I + 1>(v);
    }
}

template <int M, int PH> __device__ __forceinline__ void to_tile(float* sm, const float* v, int t) {
    using G = Small<M>;
    float* p = sm + spos(thread_base<M, PH>(t));
#pragma unroll
    for (int r = 0; r < (1 << G::K); ++r) p[spos(G::off(PH, r))] = v[r];
}
template <int M, int PH> __device__ __forceinline__ void from_tile(const float* sm, float* v, int t) {
    using G = Small<M>;
    const float* p = sm + spos(thread_base<M, PH>(t));
#pragma unroll
    for (int r = 0; r < (1 << G::K); ++r) v[r] = p[spos(G::off(PH, r))];
}

// A phase's elements are stored where they were loaded, so one barrier per
// exchange is enough.
template <int M, int PH> __device__ __forceinline__ void forward(float* sm, float* v, int t) {
    stages<M, PH>(v);
    if constexpr (PH + 1 < Small<M>::NPH) {
        to_tile<M, PH>(sm, v, t);
        __syncthreads();
        from_tile<M, PH + 1>(sm, v, t);
        forward<M, PH + 1>(sm, v, t);
    }
}
template <int M, int PH> __device__ __forceinline__ void inverse(float* sm, float* v, int t) {
    if constexpr (PH > 0) {
        to_tile<M, PH>(sm, v, t);
        __syncthreads();
        from_tile<M, PH - 1>(sm, v, t);
        stages<M, PH - 1>(v);
        inverse<M, PH - 1>(sm, v, t);
    }
}

template <int M>
__global__ void __launch_bounds__(Small<M>::NT) k2_small(SmallArgs a) {
    using G = Small<M>;
    constexpr int N = 1 << M, NT = G::NT, NE = 1 << G::K, LAST = G::NPH - 1;
    // dynamic shared memory only (the kernel's limit is set to the device maximum)
    extern __shared__ __align__(16) unsigned char smraw[];
    float* sm = reinterpret_cast<float*>(smraw);
    uint16_t* scls = reinterpret_cast<uint16_t*>(smraw + (spos(N - 1) + 4) / 4 * 16);
    double* tot = reinterpret_cast<double*>(scls + N);
    int* first = reinterpret_cast<int*>(tot + 2 * a.nb);
    float* bins = reinterpret_cast<float*>(first + 4);
    const int t = threadIdx.x, nb2 = 2 * a.nb;
    chain_begin();
    const long long fn = blockIdx.x;
    const float* src = a.f + fn * a.ld;
    float* dst = a.c + fn * a.ld;
    float v[NE], w[NE];
    {
        const float* p = src + thread_base<M, 0>(t);
#pragma unroll
        for (int r = 0; r < NE; ++r) v[r] = p[G::off(0, r)];
    }
    const int be = thread_base<M, LAST>(t);
#pragma unroll
    for (int r = 0; r < NE; ++r) w[r] = a.W ? __ldg(a.W + be + G::off(LAST, r)) : 1.f;
    if (a.nwb) {
        for (int i = t; i < N / 8; i += NT)
            reinterpret_cast<uint4*>(scls)[i] = __ldg(reinterpret_cast<const uint4*>(a.cls) + i);
        for (int i = t; i < a.nwb * nb2 * 8; i += NT) reinterpret_cast<float4*>(bins)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    forward<M, 0>(sm, v, t);
    // scale (a power of two), weight; the tile keeps g for the class sums
#pragma unroll
    for (int r = 0; r < NE; ++r) v[r] = (v[r] * a.scale) * w[r];
    if (a.coef) {
        float* g = a.coef + fn * a.ld + be;
#pragma unroll
        for (int r = 0; r < NE; ++r) g[G::off(LAST, r)] = v[r];
    }
    if (a.nwb) {
        to_tile<M, LAST>(sm, v, t);
        stages<M, LAST>(v);   // the inverse's first phase
        __syncthreads();
        if (t < a.nwb * 32) {
            const int step = a.nwb * 32;
            float* bt = bins + (t >> 5) * nb2 * 32 + (t & 31);
            float* bs = bt + a.nb * 32;
            for (int e0 = t; e0 < N; e0 += 8 * step) {
                float q[8];
                unsigned k[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int e = e0 + j * step;
                    const bool ok = e < N && e > 0;   // the label H = 0 is in no class
                    q[j] = ok ? sm[spos(e)] : 0.f;
                    k[j] = ok ? scls[e] : 0u;
                }
                // two elements at a time: their bins are loaded together; if both
                // fall in one bin the second adds to the first's sum
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    const int kt0 = (int)(k[j] & 255u), ks0 = (int)(k[j] >> 8);
                    const int kt1 = (int)(k[j + 1] & 255u), ks1 = (int)(k[j + 1] >> 8);
                    const float xt0 = bt[32 * kt0], xt1 = bt[32 * kt1], xs0 = bs[32 * ks0], xs1 = bs[32 * ks1];
                    // (a bin grows by g^2 in one rounding, as in the generic pass)
                    const float rt0 = __fmaf_rn(q[j], q[j], xt0), rs0 = __fmaf_rn(q[j], q[j], xs0);
                    const float rt1 = __fmaf_rn(q[j + 1], q[j + 1], kt1 == kt0 ? rt0 : xt1);
                    const float rs1 = __fmaf_rn(q[j + 1], q[j + 1], ks1 == ks0 ? rs0 : xs1);
                    bt[32 * kt0] = rt0;
                    bs[32 * ks0] = rs0;
                    bt[32 * kt1] = rt1;
                    bs[32 * ks1] = rs1;
                }
            }
        }
        __syncthreads();
        // four classes at a time: their trees overlap
        for (int b0 = 4 * (t >> 5); b0 < nb2; b0 += 4 * (NT / 32)) {
            float x[4] = {0.f, 0.f, 0.f, 0.f};
            for (int ww = 0; ww < a.nwb; ++ww) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (b0 + k < nb2) x[k] += bins[(ww * nb2 + b0 + k) * 32 + (t & 31)];
            }
#pragma unroll
            for (int h = 16; h > 0; h >>= 1) {
#pragma unroll
                for (int k = 0; k < 4; ++k) x[k] += __shfl_xor_sync(0xffffffffu, x[k], h);
            }
            if ((t & 31) == 0) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (b0 + k < nb2) tot[b0 + k] = (double)x[k];
            }
        }
    } else {
        stages<M, LAST>(v);
    }
    inverse<M, LAST>(sm, v, t);
    {
        float* p = dst + thread_base<M, 0>(t);
#pragma unroll
        for (int r = 0; r < NE; ++r) p[G::off(0, r)] = v[r];
    }
    if (a.nwb) {
        __syncthreads();
        effdim_outputs(tot, first, a.nb, a.thr, a.o, fn);
    }
}

template <int M> int launch_small(const SmallArgs& a, int batch, cudaStream_t st) {
    using G = Small<M>;
    auto k = k2_small<M>;
    int rc = smem_limit_max(k);
    if (rc) return rc;
    const size_t smem = (size_t)(spos((1 << M) - 1) + 4) / 4 * 16 + ((size_t)2 << M) + (size_t)2 * a.nb * 8 + 16 +
                        (size_t)a.nwb * 2 * a.nb * 128;
    {
        LaunchScope ls("interp_small", st);
        launch_chain(k, dim3((unsigned)batch), G::NT, smem, st, a);
    }
    DWT_CK_LAUNCH("k2_small");
    return DWT_OK;
}

}  // namespace

// Sizes of the one-launch form.  The upper end is the largest tile of one CTA
// (64 KB); below 2^8 points the generic pass is as fast.
bool p2_small_ok(int m) { return m >= 8 && m <= 14; }

int p2_small_interpolate(dwt_plan_s* Pl, const float* f, float* c, float* coef, int batch, long long ld,
                         bool weighted, double thr, const EffOut& o, cudaStream_t st) {
    const int m = Pl->m, nb = Pl->s + 1;
    SmallArgs a{};
    a.f = f;
    a.c = c;
    a.coef = coef;
    a.W = weighted ? Pl->d_W : nullptr;
    a.cls = Pl->d_cls;
    a.ld = ld;
    a.scale = (float)(1.0 / (double)Pl->N);
    a.nb = nb;
    // one warp per 2^10 points, within 16 warps and 48 KB of bins
    const int most = std::max(1, std::min(16, 1 << std::max(0, m - 10)));
    if (o.vt || o.vs || o.dt || o.ds) a.nwb = std::max(1, std::min(most, (48 * 1024) / (2 * nb * 128)));
    a.thr = thr;
    a.o = o;
    switch (m) {
        case 8: return launch_small<8>(a, batch, st);
        case 9: return launch_small<9>(a, batch, st);
        case 10: return launch_small<10>(a, batch, st);
        case 11: return launch_small<11>(a, batch, st);
        case 12: return launch_small<12>(a, batch, st);
        case 13: return launch_small<13>(a, batch, st);
        case 14: return launch_small<14>(a, batch, st);
        default: set_error("small interpolation: m"); return DWT_EUNSUPPORTED;
    }
}

}  // namespace dwt
