// dwt_pass.cuh -- radix-p Walsh (Chrestenson) transforms over digital nets,
// Algorithm 1 (forward, eq. fdwt) and Algorithm 2 (inverse), plus the fused
// weighting / effective-dimension pass of the interpolation (Sec. 3, Sec. 4).
//
// The transform of Sec. 2.2 is the Kronecker power over the m index digits of
// the p-point DFT F[h][n] = omega^{-hn}: the sum over digit n_r touches nothing
// but digit r, and the sums over different digits commute.  Digits are
// therefore processed in passes of b digits each; a pass covers a tile of p^b
// "rows" (one per value of its digits) times Wc "columns" (consecutive values
// of the digits below the pass).  Inside a tile every thread takes p^K elements
// that differ only in K consecutive digits and runs those K stages in
// registers; groups of K digits follow one another through shared memory, the
// first read straight from global memory and the last, where the rows allow,
// written straight back.
//
// Every prime's kernels are instantiated in a translation unit of their own
// (dwt_pass_p<P>.cu), so that they compile in parallel.
#pragma once

#include <string.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "dwt_internal.cuh"

namespace dwt {

// ---------------------------------------------------------------------------
// element helpers
struct Tw {
    float c[32], s[32];   // cos, sin of 2 pi e / p, e < p <= 31
    double cd[32], sd[32];
};

template <typename T> struct IsCplx : std::false_type {};
template <> struct IsCplx<float2> : std::true_type {};
template <> struct IsCplx<double2> : std::true_type {};

template <typename T> __device__ __forceinline__ T zero_of();
template <> __device__ __forceinline__ float zero_of<float>() { return 0.f; }
template <> __device__ __forceinline__ double zero_of<double>() { return 0.0; }
template <> __device__ __forceinline__ int zero_of<int>() { return 0; }
template <> __device__ __forceinline__ float2 zero_of<float2>() { return make_float2(0.f, 0.f); }
template <> __device__ __forceinline__ double2 zero_of<double2>() { return make_double2(0.0, 0.0); }

template <typename T, typename TI> __device__ __forceinline__ T promote(TI v) { return v; }
template <> __device__ __forceinline__ float2 promote<float2, float>(float v) { return make_float2(v, 0.f); }
template <> __device__ __forceinline__ double2 promote<double2, double>(double v) { return make_double2(v, 0.0); }

// complex FP32 on the packed f32x2 pipe: one instruction per complex add
__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) {
    unsigned long long ua, ub, ud;
    memcpy(&ua, &a, 8);
    memcpy(&ub, &b, 8);
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(ud) : "l"(ua), "l"(ub));
    float2 d;
    memcpy(&d, &ud, 8);
    return d;
}
__device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

template <typename T> __device__ __forceinline__ T scale_by(T v, double s);
template <> __device__ __forceinline__ float scale_by<float>(float v, double s) { return v * (float)s; }
template <> __device__ __forceinline__ double scale_by<double>(double v, double s) { return v * s; }
template <> __device__ __forceinline__ int scale_by<int>(int v, double) { return v; }
template <> __device__ __forceinline__ float2 scale_by<float2>(float2 v, double s) {
    return make_float2(v.x * (float)s, v.y * (float)s);
}
template <> __device__ __forceinline__ double2 scale_by<double2>(double2 v, double s) {
    return make_double2(v.x * s, v.y * s);
}

// shared-memory index with one pad element per 128 bytes (bank spreading)
template <typename T> struct PadLog { static constexpr int v = sizeof(T) == 4 ? 5 : sizeof(T) == 8 ? 4 : 3; };
template <typename T> __device__ __forceinline__ int spad(int i) { return i + (i >> PadLog<T>::v); }
template <typename T> static inline size_t spad_bytes(int nel) {
    int last = nel - 1;
    return (size_t)(last + (last >> PadLog<T>::v) + 1) * sizeof(T);
}

constexpr int cpow(int p, int k) { return k == 0 ? 1 : p * cpow(p, k - 1); }

// ---------------------------------------------------------------------------
// one p-point DFT y_t = sum_u omega^{SGN u t} x_u in registers, odd p.  The
// terms u and p - u pair up: with s_u = x_u + x_{p-u} and d_u = x_u - x_{p-u},
//   y_t     = x_0 + sum_u cos(2 pi ut/p) s_u + i SGN sum_u sin(2 pi ut/p) d_u,
//   y_{p-t} = the same with the sine sum negated,
// for u, t = 1 .. (p-1)/2: real-by-complex products only, shared by both outputs.
template <typename T> struct TwOf;
template <> struct TwOf<float2> {
    static __device__ __forceinline__ float c(const Tw& tw, int e) { return tw.c[e]; }
    static __device__ __forceinline__ float s(const Tw& tw, int e) { return tw.s[e]; }
};
template <> struct TwOf<double2> {
    static __device__ __forceinline__ double c(const Tw& tw, int e) { return tw.cd[e]; }
    static __device__ __forceinline__ double s(const Tw& tw, int e) { return tw.sd[e]; }
};

// y = c x + a for real c and complex x, a
__device__ __forceinline__ float2 cfma(float c, float2 x, float2 a) { return __ffma2_rn(make_float2(c, c), x, a); }
__device__ __forceinline__ double2 cfma(double c, double2 x, double2 a) {
    return make_double2(fma(c, x.x, a.x), fma(c, x.y, a.y));
}
// a + g i b with g = +-1: (a.x - g b.y, a.y + g b.x)
template <int G> __device__ __forceinline__ float2 add_ib(float2 a, float2 b) {
    return __ffma2_rn(make_float2(-(float)G, (float)G), make_float2(b.y, b.x), a);
}
template <int G> __device__ __forceinline__ double2 add_ib(double2 a, double2 b) {
    return make_double2(a.x - G * b.y, a.y + G * b.x);
}

template <int P, int SGN, typename T> struct Dft {
    static __device__ __forceinline__ void run(T* x, const Tw& tw) {
        static_assert(IsCplx<T>::value, "p > 2 needs complex data");
        constexpr int H = (P - 1) / 2;
        T sp[H], dm[H];
        T y0 = x[0];
#pragma unroll
        for (int u = 1; u <= H; ++u) {
            sp[u - 1] = x[u] + x[P - u];
            dm[u - 1] = x[u] - x[P - u];
            y0 = y0 + sp[u - 1];
        }
#pragma unroll
        for (int t = 1; t <= H; ++t) {
            T a = x[0], b = zero_of<T>();
#pragma unroll
            for (int u = 1; u <= H; ++u) {
                const int e = (u * t) % P;
                a = cfma(TwOf<T>::c(tw, e), sp[u - 1], a);
                b = cfma(TwOf<T>::s(tw, e), dm[u - 1], b);
            }
            x[t] = add_ib<SGN>(a, b);
            x[P - t] = add_ib<-SGN>(a, b);
        }
        x[0] = y0;
    }
};

// p = 2: omega = -1 both ways
template <int SGN, typename T> struct Dft<2, SGN, T> {
    static __device__ __forceinline__ void run(T* x, const Tw&) {
        T a = x[0], b = x[1];
        x[0] = a + b;
        x[1] = a - b;
    }
};

// K stages over the K digits of a register array of P^K elements
template <int P, int NK, int ST, int SGN, typename T> struct RegStages {
    static __device__ __forceinline__ void run(T* v, const Tw& tw) {
#pragma unroll
        for (int blk = 0; blk < NK; blk += ST * P) {
#pragma unroll
            for (int off = 0; off < ST; ++off) {
                T x[P];
#pragma unroll
                for (int u = 0; u < P; ++u) x[u] = v[blk + off + u * ST];
                Dft<P, SGN, T>::run(x, tw);
#pragma unroll
                for (int u = 0; u < P; ++u) v[blk + off + u * ST] = x[u];
            }
        }
        RegStages<P, NK, ST * P, SGN, T>::run(v, tw);
    }
};
template <int P, int NK, int SGN, typename T> struct RegStages<P, NK, NK, SGN, T> {
    static __device__ __forceinline__ void run(T*, const Tw&) {}
};

// loads and stores with an L2 eviction priority: the first pass reads its input
// for the last time and the last pass writes final results (evict first), so
// that the intermediate of the passes between stays in L2
__device__ __forceinline__ uint64_t l2_policy(int first) {
    uint64_t p;
    if (first) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    else asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ float ld_l2(const float* a, uint64_t p) {
    float v;
    asm volatile("ld.global.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(a), "l"(p));
    return v;
}
__device__ __forceinline__ int ld_l2(const int* a, uint64_t p) {
    int v;
    asm volatile("ld.global.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(v) : "l"(a), "l"(p));
    return v;
}
__device__ __forceinline__ double ld_l2(const double* a, uint64_t p) {
    double v;
    asm volatile("ld.global.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(a), "l"(p));
    return v;
}
__device__ __forceinline__ float2 ld_l2(const float2* a, uint64_t p) {
    float2 v;
    asm volatile("ld.global.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(a), "l"(p));
    return v;
}
__device__ __forceinline__ double2 ld_l2(const double2* a, uint64_t p) {
    double2 v;
    asm volatile("ld.global.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;" : "=d"(v.x), "=d"(v.y) : "l"(a), "l"(p));
    return v;
}
__device__ __forceinline__ void st_l2(float* a, float v, uint64_t p) {
    asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(a), "f"(v), "l"(p) : "memory");
}
__device__ __forceinline__ void st_l2(int* a, int v, uint64_t p) {
    asm volatile("st.global.L2::cache_hint.s32 [%0], %1, %2;" ::"l"(a), "r"(v), "l"(p) : "memory");
}
__device__ __forceinline__ void st_l2(double* a, double v, uint64_t p) {
    asm volatile("st.global.L2::cache_hint.f64 [%0], %1, %2;" ::"l"(a), "d"(v), "l"(p) : "memory");
}
__device__ __forceinline__ void st_l2(float2* a, float2 v, uint64_t p) {
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(a), "f"(v.x), "f"(v.y), "l"(p) : "memory");
}
__device__ __forceinline__ void st_l2(double2* a, double2 v, uint64_t p) {
    asm volatile("st.global.L2::cache_hint.v2.f64 [%0], {%1, %2}, %3;" ::"l"(a), "d"(v.x), "d"(v.y), "l"(p) : "memory");
}

// digits per register group: p^K elements per thread (27 complex FP32 at p = 3)
template <int P, typename T> struct KMax {
    static constexpr int v = P == 2 ? (sizeof(T) == 8 ? 4 : 5)
                                    : (sizeof(T) == 8 ? (P == 3 ? 3 : P == 5 ? 2 : 1) : (P == 3 ? 2 : 1));
};

// ---------------------------------------------------------------------------
// one register group of a pass: k digits from row digit g0 on, in the order
// they run; the divisions of the task numbering as multiplications
struct PassGroup {
    unsigned pg0, nrh;       // p^g0, R / p^(g0+k)
    unsigned mg_lo, mg_hi;   // floor(2^32 / d) + 1 for d = pg0 and nrh, 0 for d = 1
    int k, last;
};
constexpr int kMaxGroups = 8;   // 64 KB tiles: at most five (p = 5, complex FP64)

struct PassArgs {
    const void* in;
    void* out;
    long long ld_in, ld_out;
    long long S, SR;
    unsigned nlo;
    int R, Wc, wlog;
    double scale;
    float scalef;
    int do_scale;
    int direct_out;          // the last group writes global memory
    int in_first, out_first; // input read, output written for the last time
    PassGroup g[kMaxGroups];
};

// Register groups of a pass.  A tile has R = p^b rows (row digits 0 .. b-1) of
// Wc columns; element (r, c) sits at tile index (r << wlog) + c in shared
// memory and at offset c + S r from the tile base in global memory.  A group
// runs the stages of the k row digits [g0, g0 + k): each task holds the p^k
// elements that differ in those digits, rows r0 + i p^g0 with
// r0 = rl + rh p^(g0+k) (rl < p^g0, rh < R / p^(g0+k)), in one column.  Tasks
// are numbered column first, then rl, then rh, so that neighbouring threads
// touch neighbouring columns and rows (coalesced global access); with RHF the
// order of rl and rh is swapped, so that neighbouring threads are p^(g0+k)
// rows apart: an odd stride for odd p, which spreads them over all shared
// memory banks without padding.  A group reads from global memory (SRC_G) or
// shared memory and writes to global memory (DST_G) or shared memory.
template <int P, typename T> __device__ __forceinline__ int sx(int e) { return (P & 1) ? e : spad<T>(e); }

template <typename T> __device__ __forceinline__ T scale_of(const PassArgs& a, T v) {
    if constexpr (sizeof(T) == sizeof(float) || std::is_same<T, float2>::value) return scale_by<T>(v, a.scalef);
    else return scale_by<T>(v, a.scale);
}

// Everything that does not depend on the element is worked out on the host
// (PassGroup) or once per task, and an element's address is the previous one's
// plus a stride: with the divisions, products and 64-bit offsets per thread and
// element that this replaces, p = 3 spent 79 instructions per point on eight
// digits, of which the sums need 24.
template <int P, int K, int SGN, typename T, typename TI, bool SRC_G, bool DST_G, bool RHF>
__device__ __forceinline__ void rgroup(T* sm, const TI* gin, T* gout, const PassGroup& g, const PassArgs& a,
                                       const Tw& tw, int ncols) {
    constexpr int NK = cpow(P, K);
    const unsigned pg0 = g.pg0, pgk = pg0 * NK;
    const unsigned ntask = ((unsigned)a.R / NK) << a.wlog;
    // q / dv by a multiplication, exact while q dv < 2^32 (q, dv <= R <= 2^16 here)
    const unsigned dv = RHF ? g.nrh : pg0, mg = RHF ? g.mg_hi : g.mg_lo;
    const unsigned cmask = (unsigned)a.Wc - 1;
    const int sstep = (int)(pg0 << a.wlog);
    const long long gstep = a.S * (long long)pg0;
    for (unsigned t = threadIdx.x; t < ntask; t += blockDim.x) {
        const unsigned c = t & cmask, q = t >> a.wlog;
        const unsigned qd = mg ? __umulhi(q, mg) : q, qm = q - qd * dv;
        const unsigned rl = RHF ? qd : qm, rh = RHF ? qm : qd;
        const unsigned r0 = rl + rh * pgk;
        const bool live = (int)c < ncols;
        const int e0 = (int)((r0 << a.wlog) + c);
        T v[NK];
        if constexpr (SRC_G) {
            const TI* src = gin + (c + a.S * (long long)r0);
            const uint64_t pol = l2_policy(a.in_first);
#pragma unroll
            for (int i = 0; i < NK; ++i) {
                v[i] = live ? promote<T, TI>(ld_l2(src, pol)) : zero_of<T>();
                src += gstep;
            }
        } else {
            int e = e0;
#pragma unroll
            for (int i = 0; i < NK; ++i) {
                v[i] = sm[sx<P, T>(e)];
                e += sstep;
            }
        }
        RegStages<P, NK, 1, SGN, T>::run(v, tw);
        if constexpr (DST_G) {
            if (a.do_scale) {
#pragma unroll
                for (int i = 0; i < NK; ++i) v[i] = scale_of<T>(a, v[i]);
            }
            if (live) {
                T* dst = gout + (c + a.S * (long long)r0);
                const uint64_t pol = l2_policy(a.out_first);
#pragma unroll
                for (int i = 0; i < NK; ++i) {
                    st_l2(dst, v[i], pol);
                    dst += gstep;
                }
            }
        } else {
            int e = e0;
#pragma unroll
            for (int i = 0; i < NK; ++i) {
                sm[sx<P, T>(e)] = v[i];
                e += sstep;
            }
        }
    }
}

// mode bits: 1 read global, 2 write global, 4 rh-first numbering
template <int P, int SGN, typename T, typename TI, int K>
__device__ __forceinline__ void rgroup_k(int mode, T* sm, const TI* gin, T* gout, const PassGroup& g,
                                         const PassArgs& a, const Tw& tw, int ncols) {
    if constexpr (K >= 1) {
        if (g.k == K) {
            switch (mode) {
                case 1: rgroup<P, K, SGN, T, TI, true, false, false>(sm, gin, gout, g, a, tw, ncols); break;
                case 2: rgroup<P, K, SGN, T, TI, false, true, false>(sm, gin, gout, g, a, tw, ncols); break;
                case 3: rgroup<P, K, SGN, T, TI, true, true, false>(sm, gin, gout, g, a, tw, ncols); break;
                default:
                    if constexpr (P & 1) rgroup<P, K, SGN, T, TI, false, false, true>(sm, gin, gout, g, a, tw, ncols);
                    else rgroup<P, K, SGN, T, TI, false, false, false>(sm, gin, gout, g, a, tw, ncols);
                    break;
            }
            return;
        }
        rgroup_k<P, SGN, T, TI, K - 1>(mode, sm, gin, gout, g, a, tw, ncols);
    }
}

// One pass over the digits d0 .. d0+b-1 of every function: grid (tiles,
// functions).  The first group takes the top digits and reads the tile from
// global memory straight into registers (coalesced: neighbouring threads hold
// neighbouring rows, or columns); the other digits follow bottom-up through
// shared memory.  The last group, which then has the longest runs of
// neighbouring rows below it, writes straight to global memory when a run
// (p^g0 rows in the low pass, Wc columns in the others) spans at least 64
// bytes; otherwise it writes shared memory and the tile leaves in element
// order.  In place is safe: a tile is read in full before any of it is written
// (a one-group pass reads and writes the same elements per thread).
// Register cap: 96 x 512 threads fit the register file; a single digit of a
// prime above 13 holds p complex elements and the p-point sums, so those
// passes get 160 registers and at most 384 threads.
template <int P, typename T> constexpr int pass_maxnreg() {
    return P > 13 ? 160 : sizeof(T) == 8 && P == 3 ? 80 : sizeof(T) == 8 && P == 5 ? 72 : 96;
}
template <int P> constexpr long long pass_max_threads() { return P > 13 ? 384 : 512; }

template <int P, typename T, typename TI, int SGN, int KM>
__device__ __forceinline__ void pass_body(const PassArgs& a, const Tw& tw, unsigned tile, long long fn) {
    extern __shared__ __align__(16) unsigned char smraw[];
    T* sm = reinterpret_cast<T*>(smraw);
    const unsigned th = tile / a.nlo;
    const long long lo0 = (long long)(tile - th * a.nlo) << a.wlog;
    const long long base = lo0 + th * a.SR;
    const int ncols = (int)min((long long)a.Wc, a.S - lo0);
    const TI* in = reinterpret_cast<const TI*>(a.in) + fn * a.ld_in + base;
    T* out = reinterpret_cast<T*>(a.out) + fn * a.ld_out + base;
    const bool direct_out = a.direct_out != 0;
    for (int i = 0; i < kMaxGroups; ++i) {
        const PassGroup& g = a.g[i];
        const bool to_out = g.last && direct_out;
        rgroup_k<P, SGN, T, TI, KM>((i == 0 ? 1 : 0) | (to_out ? 2 : 0) | (i != 0 && !to_out ? 4 : 0), sm, in, out, g, a,
                                    tw, ncols);
        if (!to_out) __syncthreads();
        if (g.last) break;
    }
    if (!direct_out) {
        const int nel = a.R << a.wlog;
        const int cmask = a.Wc - 1;
        for (int e = threadIdx.x; e < nel; e += blockDim.x) {
            const int r = e >> a.wlog, c = e & cmask;
            if (c < ncols) {
                T v = sm[sx<P, T>(e)];
                if (a.do_scale) v = scale_of<T>(a, v);
                out[c + (long long)r * a.S] = v;
            }
        }
    }
}

template <int P, typename T, typename TI, int SGN, int KM>
__global__ void __maxnreg__((pass_maxnreg<P, T>())) k_pass(PassArgs a, const __grid_constant__ Tw tw) {
    chain_begin();
    pass_body<P, T, TI, SGN, KM>(a, tw, blockIdx.x, blockIdx.y);
}

// One pass of several plans' transforms in one launch: job i owns the blocks
// [first, first + ntile * nf) (tile fastest).  Each block runs exactly the tile
// body of k_pass, so every element is computed as by the plan's own launch.
// Lists of up to kGroupInline jobs travel in the launch's parameters; longer
// ones lie in device memory.  (An allocation and a copy per launch cost more
// host time than the launch: 8 jobs of 2^8 .. 2^15 points in five launches,
// 49 us per call with them, 26 us without.)
struct GroupPass {
    PassArgs a;
    long long ntile, first;
};
constexpr int kGroupInline = 32;
struct GroupList {
    Tw tw;
    int n;
    const GroupPass* far;   // n > kGroupInline
    GroupPass near[kGroupInline];
};

template <int P, typename T, typename TI, int SGN, int KM>
__global__ void __maxnreg__(P > 13 ? 160 : 96) k_pass_grouped(const __grid_constant__ GroupList list) {
    chain_begin();
    const GroupPass* jobs = list.n > kGroupInline ? list.far : list.near;
    const long long b = blockIdx.x;
    int lo = 0, hi = list.n - 1;   // the last job starting at or before b
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].first <= b) lo = mid;
        else hi = mid - 1;
    }
    const GroupPass& g = jobs[lo];
    const unsigned local = (unsigned)(b - g.first), fn = local / (unsigned)g.ntile;
    pass_body<P, T, TI, SGN, KM>(g.a, list.tw, local - fn * (unsigned)g.ntile, fn);
}

// ---------------------------------------------------------------------------
// fused top pass of the interpolation: forward stages of the last digits,
// scale p^-m, weight, per-class variance partials, optional coefficient store,
// inverse stages of the same digits.
struct MidArgs {
    PassArgs pa;
    const float* W;        // NULL: weight 1
    const uint8_t* cls;    // [N][2]
    void* coef;            // optional output of g
    double* part;          // [fn][ntile][2*nb]
    long long ntile;
    int nb;                // s + 1
};

template <typename T> __device__ __forceinline__ float mag2(T v);
template <> __device__ __forceinline__ float mag2<float>(float v) { return v * v; }
template <> __device__ __forceinline__ float mag2<float2>(float2 v) { return v.x * v.x + v.y * v.y; }
// bin + |v|^2: one rounding for real v (a fused multiply-add)
template <typename T> __device__ __forceinline__ float add_mag2(float bin, T v);
template <> __device__ __forceinline__ float add_mag2<float>(float bin, float v) { return __fmaf_rn(v, v, bin); }
template <> __device__ __forceinline__ float add_mag2<float2>(float bin, float2 v) { return bin + mag2<float2>(v); }
template <typename T> __device__ __forceinline__ T mulw(T v, float w);
template <> __device__ __forceinline__ float mulw<float>(float v, float w) { return v * w; }
template <> __device__ __forceinline__ float2 mulw<float2>(float2 v, float w) { return make_float2(v.x * w, v.y * w); }

// per-lane FP32 class sums of the first nwb warps -> one FP64 value per class
// and tile, fixed order
__device__ __forceinline__ void reduce_bins(const float* bins, int nb2, int nwb, double* out, long long stride) {
    // four classes at a time: their trees overlap
    const int nw = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int b0 = 4 * w; b0 < nb2; b0 += 4 * nw) {
        float x[4] = {0.f, 0.f, 0.f, 0.f};
        for (int ww = 0; ww < nwb; ++ww) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (b0 + k < nb2) x[k] += bins[(ww * nb2 + b0 + k) * 32 + lane];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] += __shfl_xor_sync(0xffffffffu, x[k], o);
        }
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (b0 + k < nb2) out[(b0 + k) * stride] = (double)x[k];
        }
    }
}

// The fused top pass in register groups (as k_pass): forward groups from the
// top digits down, the last one leaving the tile in shared memory; the scale,
// weight, optional coefficient store and class partials (per-lane FP32 bins of
// the first nwb warps, a fixed summation order) element by element; then the
// inverse groups, the last one writing global memory as in k_pass.
template <int P, typename T, typename TI, int KM>
__global__ void __maxnreg__(96) k_mid(MidArgs m, int nwb, const __grid_constant__ Tw tw) {
    chain_begin();
    const PassArgs& a = m.pa;
    extern __shared__ __align__(16) unsigned char smraw[];
    T* sm = reinterpret_cast<T*>(smraw);
    const int nel = a.R << a.wlog;
    const int tile_elems = nel + ((nel - 1) >> PadLog<T>::v);   // as spad_bytes on the host
    float* bins = reinterpret_cast<float*>(smraw + ((tile_elems * sizeof(T) + 15) & ~(size_t)15));
    const int nb2 = 2 * m.nb;
    const long long fn = blockIdx.y;
    const unsigned tile = blockIdx.x, th = tile / a.nlo;
    const long long lo0 = (long long)(tile - th * a.nlo) << a.wlog;
    const long long base = lo0 + th * a.SR;
    const int ncols = (int)min((long long)a.Wc, a.S - lo0);
    const int cmask = a.Wc - 1;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const TI* in = reinterpret_cast<const TI*>(a.in) + fn * a.ld_in + base;
    T* out = reinterpret_cast<T*>(a.out) + fn * a.ld_out + base;
    for (int i = threadIdx.x; i < nwb * nb2 * 8; i += blockDim.x)
        reinterpret_cast<float4*>(bins)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool direct_out = a.direct_out != 0;
    // forward stages
    for (int i = 0; i < kMaxGroups; ++i) {
        const PassGroup& g = a.g[i];
        rgroup_k<P, -1, T, TI, KM>(i == 0 ? 1 : 4, sm, in, out, g, a, tw, ncols);
        __syncthreads();
        if (g.last) break;
    }
    // scale, weight, coefficients, class partials: lane l of warp w < nwb takes the
    // elements 32 w + l, + 32 nwb, ... in order, eight at a time with the next
    // eight's weights and classes on their way (p = 3, m = 13, 3 functions: 38.6 ->
    // 35.2 us).  Labels fit 32 bits (N <= 2^31).  Two
    // elements' bins are loaded together and stored together; if both fall in one
    // bin the second adds to the first's sum.
    if (w < nwb) {
        float* bt = bins + (size_t)w * nb2 * 32 + lane;
        float* bs = bt + m.nb * 32;
        T* coef = m.coef ? reinterpret_cast<T*>(m.coef) + fn * a.ld_out : nullptr;
        const int step = nwb * 32;
        const unsigned S = (unsigned)a.S, base32 = (unsigned)base;
        float wn[8];
        unsigned kn[8];
        auto label = [&](int e) {   // 0 past the tile or its columns
            const int r = e >> a.wlog, c = e & cmask;
            return e < nel && c < ncols ? base32 + (unsigned)c + (unsigned)r * S : 0u;
        };
        auto load = [&](int e0) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const unsigned H = label(e0 + j * step);
                wn[j] = m.W ? __ldg(m.W + H) : 1.f;
                kn[j] = __ldg(reinterpret_cast<const unsigned short*>(m.cls) + H);
            }
        };
        load(threadIdx.x);
        for (int e0 = threadIdx.x; e0 < nel; e0 += 8 * step) {
            float wv[8];
            unsigned kc[8], H[8];
            bool ok[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int e = e0 + j * step;
                ok[j] = e < nel && (e & cmask) < ncols;
                H[j] = label(e);
                wv[j] = wn[j];
                kc[j] = kn[j];
            }
            if (e0 + 8 * step < nel) load(e0 + 8 * step);   // in flight during this round's bins
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                T q[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    q[u] = zero_of<T>();   // the label H = 0 is in no class
                    if (ok[j + u]) {
                        T& x = sm[sx<P, T>(e0 + (j + u) * step)];
                        const T v = mulw<T>(scale_of<T>(a, x), wv[j + u]);
                        x = v;
                        if (coef) coef[H[j + u]] = v;
                        if (H[j + u] != 0) q[u] = v;
                    }
                }
                const int kt0 = (int)(kc[j] & 255u), ks0 = (int)(kc[j] >> 8);
                const int kt1 = (int)(kc[j + 1] & 255u), ks1 = (int)(kc[j + 1] >> 8);
                const float xt0 = bt[32 * kt0], xt1 = bt[32 * kt1], xs0 = bs[32 * ks0], xs1 = bs[32 * ks1];
                const float rt0 = add_mag2<T>(xt0, q[0]), rs0 = add_mag2<T>(xs0, q[0]);
                const float rt1 = add_mag2<T>(kt1 == kt0 ? rt0 : xt1, q[1]), rs1 = add_mag2<T>(ks1 == ks0 ? rs0 : xs1, q[1]);
                bt[32 * kt0] = rt0;
                bs[32 * ks0] = rs0;
                bt[32 * kt1] = rt1;
                bs[32 * ks1] = rs1;
            }
        }
    }
    __syncthreads();
    reduce_bins(bins, nb2, nwb, m.part + fn * nb2 * m.ntile + tile, m.ntile);
    // inverse stages of the same digits, in the same order
    for (int i = 0; i < kMaxGroups; ++i) {
        const PassGroup& g = a.g[i];
        const bool dst_g = g.last && direct_out;
        rgroup_k<P, +1, T, T, KM>(dst_g ? 2 : 4, sm, out, out, g, a, tw, ncols);
        if (!dst_g) __syncthreads();
        if (g.last) break;
    }
    if (!direct_out) {
        for (int e = threadIdx.x; e < nel; e += blockDim.x) {
            const int r = e >> a.wlog, c = e & cmask;
            if (c < ncols) out[c + (long long)r * a.S] = sm[sx<P, T>(e)];
        }
    }
}
// ---------------------------------------------------------------------------
// host side
static Tw make_tw(int p) {
    Tw t;
    for (int e = 0; e < 32; ++e) {
        double ang = e < p ? 2.0 * 3.14159265358979323846 * e / p : 0.0;
        t.cd[e] = cos(ang);
        t.sd[e] = sin(ang);
        if (e == 0) { t.cd[e] = 1.0; t.sd[e] = 0.0; }
        t.c[e] = (float)t.cd[e];
        t.s[e] = (float)t.sd[e];
    }
    return t;
}

template <typename F>
static int set_smem(F* kern, size_t bytes) {
    (void)bytes;
    return smem_limit_max(kern);
}

// geometry of one pass with register groups of at most km digits: the top
// group first, then from the lowest digit up
static PassArgs pass_args(int p, int km, int elem, const PassGeom& g, const void* in, void* out, long long ld_in,
                          long long ld_out) {
    PassArgs a;
    a.in = in;
    a.out = out;
    a.ld_in = ld_in;
    a.ld_out = ld_out;
    a.S = g.S;
    a.SR = g.S * g.R;
    a.nlo = (unsigned)g.nlo;
    a.R = g.R;
    a.Wc = g.Wc;
    a.wlog = g.wlog;
    a.scale = 1.0;
    a.scalef = 1.f;
    a.do_scale = 0;
    a.in_first = a.out_first = 0;
    const int k0 = std::min(km, g.b);
    int g0 = g.b - k0, k = k0, g_last = 0;
    for (int i = 0; i < kMaxGroups; ++i) {
        PassGroup& x = a.g[i];
        x.k = k;
        x.pg0 = (unsigned)ipow_ll(p, g0);
        x.nrh = (unsigned)(g.R / ipow_ll(p, g0 + k));
        x.mg_lo = x.pg0 == 1 ? 0u : (unsigned)((1ull << 32) / x.pg0 + 1);
        x.mg_hi = x.nrh == 1 ? 0u : (unsigned)((1ull << 32) / x.nrh + 1);
        g_last = g0;
        const int next = i == 0 ? 0 : g0 + k;
        x.last = next >= g.b - k0;
        if (x.last) break;
        g0 = next;
        k = std::min(km, g.b - k0 - g0);
    }
    // a run of neighbouring elements below the last group (p^g0 rows in the low
    // pass, Wc columns in the others) of at least 64 bytes
    const long long run = g.S == 1 ? ipow_ll(p, g_last) : g.Wc;
    a.direct_out = run * elem >= 64;
    return a;
}

static void pass_scale(PassArgs& a, double scale) {
    a.do_scale = 1;
    a.scale = scale;
    a.scalef = (float)scale;
}

// L2 priorities of pass t of q: the first pass reads its input, the last pass its
// intermediate for the last time and writes final results
static void pass_ends(PassArgs& a, int t, int q) {
    a.in_first = t == 0 || t == q - 1;
    a.out_first = t == q - 1;
}

// the fused top pass of an interpolation: the only pass, or between two others
// (its results are read again by the inverse passes)
static PassArgs mid_pass_args(int p, int km, int elem, const PassPlan& pp, const void* in, void* out, long long ld) {
    PassArgs a = pass_args(p, km, elem, pp.g[pp.q - 1], in, out, ld, ld);
    if (pp.q == 1) pass_ends(a, 0, 1);
    return a;
}

static const char* pass_family(int t, int q) { return t == 0 ? "pass_lo" : (t == q - 1 ? "pass_hi" : "pass_mid"); }

// threads of a pass: one per task of its first (top) group, 32 .. 512
template <int P, int KM>
static int pass_threads(const PassGeom& g) {
    const int k0 = std::min(KM, g.b);
    long long tasks = ((long long)g.R / ipow_ll(P, k0)) << g.wlog;
    tasks = (tasks + 31) / 32 * 32;
    return (int)std::min(pass_max_threads<P>(), std::max(32ll, tasks));
}

template <int P, typename T, typename TI, int SGN, int KM>
static int launch_pass_k(const PassGeom& g, const PassArgs& a, const Tw& tw, int nf, const char* fam, cudaStream_t st) {
    const size_t smem = spad_bytes<T>(g.R << g.wlog);
    auto kern = k_pass<P, T, TI, SGN, KM>;
    int rc = set_smem(kern, smem);
    if (rc) return rc;
    dim3 grid((unsigned)g.ntile, (unsigned)nf);
    {
        LaunchScope ls(fam, st);
        launch_chain(kern, grid, pass_threads<P, KM>(g), smem, st, a, tw);
    }
    DWT_CK_LAUNCH("k_pass");
    return DWT_OK;
}

template <int P, typename T, typename TI, int SGN>
static int launch_pass(const PassGeom& g, const PassArgs& a, const Tw& tw, int nf, const char* fam,
                       cudaStream_t st) {
    return launch_pass_k<P, T, TI, SGN, KMax<P, T>::v>(g, a, tw, nf, fam, st);
}

// L2-sized groups of functions: the passes of one group run back to back so
// that the intermediate stays in the 126 MB L2 between passes (kept there by the
// eviction priorities of the first and last pass).  Groups of a batch are
// equally large, so that none ends with launches of few blocks.  48 / 64 / 96 /
// 128 MB: p = 5, m = 9, 32 forward transforms 403 / 385 / 374 / 384 us; p = 3,
// m = 13, 32 299 / 272 / 257 / 253; m = 14, 16 494 / 494 / 430 / 435; p = 7,
// m = 7, 32 215 / 208 / 204 / 203.
static const long long kL2Group = 96ll << 20;

static int functions_per_group(long long bytes, long long fbytes, int batch) {
    const long long g = std::min(65535ll, std::max(1ll, bytes / fbytes));
    const long long n = (batch + g - 1) / g;
    return (int)((batch + n - 1) / n);
}

template <int P, typename T, typename TI, int SGN>
static int transform_pp(dwt_plan_s* Pl, const PassPlan& pp, double scale_by_n, const void* in, void* out, int batch,
                        long long ld_in, long long ld_out, cudaStream_t st);

template <int P, typename T, typename TI, int SGN>
static int transform_t(dwt_plan_s* Pl, const void* in, void* out, int batch, long long ld_in, long long ld_out,
                       cudaStream_t st) {
    return transform_pp<P, T, TI, SGN>(Pl, pass_plan(Pl, sizeof(T)), 1.0 / (double)Pl->N, in, out, batch, ld_in,
                                       ld_out, st);
}

// The passes of pp over a batch; a forward (SGN < 0, not int32) scales by
// scale_by_n in its last pass.
template <int P, typename T, typename TI, int SGN>
static int transform_pp(dwt_plan_s* Pl, const PassPlan& pp, double scale_by_n, const void* in, void* out, int batch,
                        long long ld_in, long long ld_out, cudaStream_t st) {
    static const Tw tw = make_tw(P);
    const long long fbytes = Pl->N * (long long)sizeof(T);
    const int G = functions_per_group(Pl->tuned_group_bytes > 0 ? Pl->tuned_group_bytes : kL2Group, fbytes, batch);
    const bool scale = SGN < 0 && !std::is_same<T, int>::value;
    for (int f0 = 0; f0 < batch; f0 += G) {
        const int nf = std::min(G, batch - f0);
        for (int t = 0; t < pp.q; ++t) {
            const PassGeom& g = pp.g[t];
            int rc;
            if (t == 0) {
                PassArgs a = pass_args(P, KMax<P, T>::v, (int)sizeof(T), g, (const TI*)in + (long long)f0 * ld_in, (T*)out + (long long)f0 * ld_out,
                                       ld_in, ld_out);
                if (scale && pp.q == 1) pass_scale(a, scale_by_n);
                pass_ends(a, t, pp.q);
                rc = launch_pass<P, T, TI, SGN>(g, a, tw, nf, pass_family(t, pp.q), st);
            } else {
                PassArgs a = pass_args(P, KMax<P, T>::v, (int)sizeof(T), g, (const T*)out + (long long)f0 * ld_out, (T*)out + (long long)f0 * ld_out,
                                       ld_out, ld_out);
                if (scale && t == pp.q - 1) pass_scale(a, scale_by_n);
                pass_ends(a, t, pp.q);
                rc = launch_pass<P, T, T, SGN>(g, a, tw, nf, pass_family(t, pp.q), st);
            }
            if (rc) return rc;
        }
    }
    return DWT_OK;
}

template <int P>
int transform_p(dwt_plan_s* Pl, const void* in, void* out, int batch, long long ld_in, long long ld_out,
                       dwt_dtype in_t, dwt_dtype out_t, int sgn, cudaStream_t st) {
    if constexpr (P == 2) {
        if (in_t == DWT_F32)
            return sgn < 0 ? transform_t<2, float, float, -1>(Pl, in, out, batch, ld_in, ld_out, st)
                           : transform_t<2, float, float, +1>(Pl, in, out, batch, ld_in, ld_out, st);
        if (in_t == DWT_F64)
            return sgn < 0 ? transform_t<2, double, double, -1>(Pl, in, out, batch, ld_in, ld_out, st)
                           : transform_t<2, double, double, +1>(Pl, in, out, batch, ld_in, ld_out, st);
        return sgn < 0 ? transform_t<2, int, int, -1>(Pl, in, out, batch, ld_in, ld_out, st)
                       : transform_t<2, int, int, +1>(Pl, in, out, batch, ld_in, ld_out, st);
    } else {
        if (out_t == DWT_C64) {
            if (sgn < 0)
                return in_t == DWT_F32 ? transform_t<P, float2, float, -1>(Pl, in, out, batch, ld_in, ld_out, st)
                                       : transform_t<P, float2, float2, -1>(Pl, in, out, batch, ld_in, ld_out, st);
            return transform_t<P, float2, float2, +1>(Pl, in, out, batch, ld_in, ld_out, st);
        }
        if (sgn < 0)
            return in_t == DWT_F64 ? transform_t<P, double2, double, -1>(Pl, in, out, batch, ld_in, ld_out, st)
                                   : transform_t<P, double2, double2, -1>(Pl, in, out, batch, ld_in, ld_out, st);
        return transform_t<P, double2, double2, +1>(Pl, in, out, batch, ld_in, ld_out, st);
    }
}

// Stages of the digits d0 .. d0+nd-1 (generic passes), forward scaled by p^-nd.
template <int P>
int digits_p(dwt_plan_s* Pl, const void* in, void* out, int batch, long long ld_in, long long ld_out,
                    dwt_dtype in_t, dwt_dtype out_t, int d0, int nd, int sgn, cudaStream_t st) {
    auto go = [&](auto tag_t, auto tag_i, auto sgn_c) {
        using T = decltype(tag_t);
        using TI = decltype(tag_i);
        constexpr int SG = decltype(sgn_c)::value;
        PassPlan pp;
        pass_plan_range(P, Pl->m, (int)sizeof(T), d0, nd, Pl->min_tiles, pp);
        return transform_pp<P, T, TI, SG>(Pl, pp, 1.0 / (double)ipow_ll(P, nd), in, out, batch, ld_in, ld_out, st);
    };
    using M = std::integral_constant<int, -1>;
    using Pp = std::integral_constant<int, +1>;
    if constexpr (P == 2) {
        if (in_t == DWT_F32) return sgn < 0 ? go(float(), float(), M()) : go(float(), float(), Pp());
        if (in_t == DWT_F64) return sgn < 0 ? go(double(), double(), M()) : go(double(), double(), Pp());
        return sgn < 0 ? go(int(), int(), M()) : go(int(), int(), Pp());
    } else {
        if (out_t == DWT_C64) {
            if (sgn < 0) return in_t == DWT_F32 ? go(float2(), float(), M()) : go(float2(), float2(), M());
            return go(float2(), float2(), Pp());
        }
        if (sgn < 0) return in_t == DWT_F64 ? go(double2(), double(), M()) : go(double2(), double2(), M());
        return go(double2(), double2(), Pp());
    }
}
// ---------------------------------------------------------------------------
// grouped transforms: pass t of every job in one launch of k_pass_grouped

template <int P, typename T, typename TI, int SGN>
static int launch_grouped(const std::vector<GroupPass>& h, const Tw& tw, long long blocks, int threads, size_t smem,
                          const char* fam, cudaStream_t st) {
    if (h.empty()) return DWT_OK;
    if (blocks > 0x7fffffffll) {
        set_error("grouped pass: %lld blocks exceed one launch", blocks);
        return DWT_EINVAL;
    }
    constexpr int KM = KMax<P, T>::v;
    auto kern = k_pass_grouped<P, T, TI, SGN, KM>;
    int rc = set_smem(kern, smem);
    if (rc) return rc;
    GroupList list;
    list.tw = tw;
    list.n = (int)h.size();
    GroupPass* d = nullptr;
    if (list.n > kGroupInline) {
        if (dmalloc((void**)&d, sizeof(GroupPass) * h.size(), st)) return DWT_ENOMEM;
        DWT_CK(cudaMemcpyAsync(d, h.data(), sizeof(GroupPass) * h.size(), cudaMemcpyHostToDevice, st));
    } else {
        std::copy(h.begin(), h.end(), list.near);
    }
    list.far = d;
    {
        LaunchScope ls(fam, st);
        launch_chain(kern, dim3((unsigned)blocks), threads, smem, st, list);
    }
    dfree(d, st);
    DWT_CK_LAUNCH("k_pass_grouped");
    return DWT_OK;
}

// pass t of the jobs (those that have one): the tiles of the launch, their number,
// and the threads and shared memory of the largest
struct GroupLaunch {
    std::vector<GroupPass> h;
    long long blocks = 0;
    int threads = 32;
    size_t smem = 0;
};
template <int P, typename T>
static GroupLaunch group_launch(const std::vector<GroupJob>& js, const std::vector<const PassPlan*>& pps, int t, bool scale) {
    constexpr int KM = KMax<P, T>::v;
    GroupLaunch l;
    for (size_t i = 0; i < js.size(); ++i) {
        const PassPlan& pp = *pps[i];
        const GroupJob& j = js[i];
        if (t >= pp.q || j.batch <= 0) continue;
        const PassGeom& g = pp.g[t];
        GroupPass gp;
        gp.a = pass_args(P, KM, (int)sizeof(T), g, t == 0 ? j.in : j.out, j.out, t == 0 ? j.ld_in : j.ld_out, j.ld_out);
        if (scale && t == pp.q - 1) pass_scale(gp.a, 1.0 / (double)j.plan->N);
        pass_ends(gp.a, t, pp.q);
        gp.ntile = g.ntile;
        gp.first = l.blocks;
        l.blocks += g.ntile * (long long)j.batch;
        l.h.push_back(gp);
        l.threads = std::max(l.threads, pass_threads<P, KM>(g));
        l.smem = std::max(l.smem, spad_bytes<T>(g.R << g.wlog));
    }
    return l;
}

// The jobs' transforms by their plans' pass plans, pass t of all jobs in one
// launch; the same tile body, geometry and scaling as transform_pp, so every
// element equals the one of the job's own call.
template <int P, typename T, typename TI, int SGN>
static int grouped_t(const std::vector<GroupJob>& js, cudaStream_t st) {
    static const Tw tw = make_tw(P);
    const bool scale = SGN < 0 && !std::is_same<T, int>::value;
    std::vector<const PassPlan*> pps;
    int qmax = 0;
    for (const GroupJob& j : js) {
        pps.push_back(&pass_plan(j.plan, sizeof(T)));
        qmax = std::max(qmax, pps.back()->q);
    }
    for (int t = 0; t < qmax; ++t) {
        const GroupLaunch l = group_launch<P, T>(js, pps, t, scale);
        const int rc = t == 0 ? launch_grouped<P, T, TI, SGN>(l.h, tw, l.blocks, l.threads, l.smem, "grouped_pass", st)
                              : launch_grouped<P, T, T, SGN>(l.h, tw, l.blocks, l.threads, l.smem, "grouped_pass", st);
        if (rc) return rc;
    }
    return DWT_OK;
}

template <int P>
int grouped_p(const std::vector<GroupJob>& js, dwt_dtype in_t, dwt_dtype out_t, int sgn, cudaStream_t st) {
    if constexpr (P == 2) {
        if (in_t == DWT_F32)
            return sgn < 0 ? grouped_t<2, float, float, -1>(js, st) : grouped_t<2, float, float, +1>(js, st);
        if (in_t == DWT_F64)
            return sgn < 0 ? grouped_t<2, double, double, -1>(js, st) : grouped_t<2, double, double, +1>(js, st);
        return sgn < 0 ? grouped_t<2, int, int, -1>(js, st) : grouped_t<2, int, int, +1>(js, st);
    } else {
        if (out_t == DWT_C64) {
            if (sgn < 0)
                return in_t == DWT_F32 ? grouped_t<P, float2, float, -1>(js, st)
                                       : grouped_t<P, float2, float2, -1>(js, st);
            return grouped_t<P, float2, float2, +1>(js, st);
        }
        if (sgn < 0)
            return in_t == DWT_F64 ? grouped_t<P, double2, double, -1>(js, st)
                                   : grouped_t<P, double2, double2, -1>(js, st);
        return grouped_t<P, double2, double2, +1>(js, st);
    }
}
// ---------------------------------------------------------------------------
// warps that keep class bins next to a tile: up to maxw within `budget` bytes
// of bins (at least one while it fits beside the tile)
static int bins_warps(size_t tile_bytes, int nb2, size_t budget = 227 * 1024, int maxw = 8) {
    const size_t avail = 227 * 1024 - ((tile_bytes + 15) & ~(size_t)15);
    const size_t per_warp = (size_t)nb2 * 32 * 4;
    if (per_warp > avail) return 0;
    return (int)std::max<size_t>(1, std::min<size_t>(maxw, std::min(avail, budget) / per_warp));
}

template <int P, typename T, typename TI>
static int interpolate_t(dwt_plan_s* Pl, const void* f, void* c, void* coef, int batch, long long ld,
                         dwt_weight weight, double* var, int* dim, double thr, cudaStream_t st) {
    const PassPlan& pp = pass_plan(Pl, sizeof(T));
    static const Tw tw = make_tw(P);
    const int nb = Pl->s + 1, nb2 = 2 * nb;
    const PassGeom& gm = pp.g[pp.q - 1];
    const long long ntile = gm.ntile;
    constexpr int KM = KMax<P, T>::v;
    const size_t tile_bytes = spad_bytes<T>(gm.R << gm.wlog);
    const int nt = pass_threads<P, KM>(gm);
    // warps that bin: their bins within 48 KB, so that the tile and its bins
    // leave room for a second CTA
    const int nw = std::min(nt / 32, bins_warps(tile_bytes, nb2, 48 * 1024, 16));
    if (nw < 1) {
        set_error("s = %d too large for the fused variance pass", Pl->s);
        return DWT_EUNSUPPORTED;
    }
    const size_t smem = ((tile_bytes + 15) & ~(size_t)15) + (size_t)nw * nb2 * 32 * 4;
    int rc = ensure_workspace(Pl, (size_t)batch * ntile * nb2 * sizeof(double), st);
    if (rc) return rc;
    double* part = (double*)Pl->d_ws;
    auto kmid_first = k_mid<P, T, TI, KM>;   // single pass: reads f directly
    auto kmid_next = k_mid<P, T, T, KM>;     // after lower passes: in place on c
    rc = set_smem(kmid_first, smem);
    if (rc) return rc;
    rc = set_smem(kmid_next, smem);
    if (rc) return rc;
    const long long fbytes = Pl->N * (long long)sizeof(T);
    const int G = functions_per_group(kL2Group, fbytes, batch);
    for (int f0 = 0; f0 < batch; f0 += G) {
        const int nf = std::min(G, batch - f0);
        const long long off = (long long)f0 * ld;
        // forward passes below the top one: f -> c
        for (int t = 0; t + 1 < pp.q; ++t) {
            const PassGeom& g = pp.g[t];
            if (t == 0) {
                PassArgs a = pass_args(P, KMax<P, T>::v, (int)sizeof(T), g, (const TI*)f + off, (T*)c + off, ld, ld);
                a.in_first = 1;
                rc = launch_pass<P, T, TI, -1>(g, a, tw, nf, "interp_fwd", st);
            } else {
                PassArgs a = pass_args(P, KMax<P, T>::v, (int)sizeof(T), g, (const T*)c + off, (T*)c + off, ld, ld);
                rc = launch_pass<P, T, T, -1>(g, a, tw, nf, "interp_fwd", st);
            }
            if (rc) return rc;
        }
        // fused top pass
        MidArgs m;
        m.pa = mid_pass_args(P, KM, (int)sizeof(T), pp, pp.q == 1 ? (const void*)((const TI*)f + off) : (const T*)c + off,
                             (T*)c + off, ld);
        m.pa.scale = 1.0 / (double)Pl->N;
        m.pa.scalef = (float)m.pa.scale;
        m.W = weight == DWT_WEIGHT_INV_SQ_WAVENUMBER ? Pl->d_W : nullptr;
        m.cls = Pl->d_cls;
        m.coef = coef ? (void*)((T*)coef + off) : nullptr;
        m.part = part + (long long)f0 * ntile * nb2;   // [fn][class][tile] of this group
        m.ntile = ntile;
        m.nb = nb;
        {
            LaunchScope ls("interp_top", st);
            dim3 grid((unsigned)ntile, (unsigned)nf);
            if (pp.q == 1) launch_chain(kmid_first, grid, nt, smem, st, m, nw, tw);
            else launch_chain(kmid_next, grid, nt, smem, st, m, nw, tw);
        }
        DWT_CK_LAUNCH("k_mid");
        // inverse passes below the top one, in place on c
        for (int t = pp.q - 2; t >= 0; --t) {
            const PassGeom& g = pp.g[t];
            PassArgs a = pass_args(P, KMax<P, T>::v, (int)sizeof(T), g, (const T*)c + off, (T*)c + off, ld, ld);
            a.in_first = a.out_first = t == 0;
            rc = launch_pass<P, T, T, +1>(g, a, tw, nf, "interp_inv", st);
            if (rc) return rc;
        }
    }
    return effdim_reduce(part, ntile, nb, batch, thr, eff_packed(var, dim, nb), st);
}

template <int P>
int interpolate_p(dwt_plan_s* Pl, const void* f, void* c, void* coef, int batch, long long ld, dwt_dtype f_t,
                  dwt_weight weight, double* var, int* dim, double thr, cudaStream_t st) {
    if constexpr (P == 2) {
        return interpolate_t<2, float, float>(Pl, f, c, coef, batch, ld, weight, var, dim, thr, st);
    } else {
        return f_t == DWT_F32
                   ? interpolate_t<P, float2, float>(Pl, f, c, coef, batch, ld, weight, var, dim, thr, st)
                   : interpolate_t<P, float2, float2>(Pl, f, c, coef, batch, ld, weight, var, dim, thr, st);
    }
}

#define DWT_INSTANTIATE_PRIME(P)                                                                                   \
    template int transform_p<P>(dwt_plan_s*, const void*, void*, int, long long, long long, dwt_dtype, dwt_dtype,  \
                                int, cudaStream_t);                                                                \
    template int digits_p<P>(dwt_plan_s*, const void*, void*, int, long long, long long, dwt_dtype, dwt_dtype,     \
                             int, int, int, cudaStream_t);                                                         \
    template int grouped_p<P>(const std::vector<GroupJob>&, dwt_dtype, dwt_dtype, int, cudaStream_t);              \
    template int interpolate_p<P>(dwt_plan_s*, const void*, void*, void*, int, long long, dwt_dtype, dwt_weight,   \
                                  double*, int*, double, cudaStream_t);

}  // namespace dwt
