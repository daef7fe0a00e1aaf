// dwt_spline.cu -- the kernel spline of Sec. 3.1 and the variances of its
// ANOVA effects (Sec. 4), in FP64.
//
// The reproducing kernel K(x, y) = prod_j (1 + gamma_j K'(x_j (-) y_j, 0)) has
// Walsh coefficients supported on all wavenumbers, and its data at the net
// points aliases them onto the cosets: K~(H) = DWT of (K(x_n, 0))_n.  The
// interpolation conditions f(x_n) = sum_v c_v K(x_n (-) x_v, 0) are diagonal
// in the Walsh basis (eq. splinecoef): c~(H) = f~(H) / (p^m K~(H)), and
// c = FIWT(c~) (Algorithm 2).  With R'(x, 0) = int K'(t, x) K'(t, 0) dt and
// R_d = prod_{j <= d} (1 + gamma_j^2 R'), eq. sig2sfu summed over the nonempty
// u within 1..d gives
//     sigma^2_trc(d) = p^{2m} sum_H |c~(H)|^2 (R~_d(H) - [H = 0]),
// and over |u| = j the degree-j part E_j = sum_{|u| = j} gamma_u^2 R_u of
// R_s = prod_j (1 + gamma_j^2 R'), built point by point with the recurrence
// of elementary symmetric polynomials, gives
//     sigma^2_sup(d) = p^{2m} sum_H |c~(H)|^2 sum_{j <= d} E~_j(H).
// The constant effect (u = {}, the squared mean) is not a variance and is
// left out; the K' and R' values come from their short forms (Sec. 4).
//
// dwt_spline_prepare builds, once per (alpha, gamma), the kernel data at the
// net points, its 1 + 2s DWTs, and keeps W_K = 1 / (p^m K~) and the 2s
// variance tables (real parts: the kernels are real and symmetric, so their
// DWTs are real up to rounding).  dwt_spline then transforms each function,
// multiplies by W_K, contracts |c~|^2 with the tables in a fixed summation
// order, and transforms back.
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "dwt_effdim.cuh"

namespace dwt {

namespace {

constexpr int kSplineMaxS = 64;
constexpr int kDotTile = 4096;   // points per block of the hold-out error

// kernel data at point n: K, R_1..R_s, E_1..E_s (rows of `out`, ld N)
__global__ void k_spline_data(const uint32_t* __restrict__ Y, long long N, int s, int p, int m,
                              const double* __restrict__ kp, const double* __restrict__ rp,
                              const double* __restrict__ gam, double* out) {
    double e[kSplineMaxS + 1];
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N; n += (long long)gridDim.x * blockDim.x) {
        double kv = 1.0, rv = 1.0;
        e[0] = 1.0;
        for (int q = 1; q <= s; ++q) e[q] = 0.0;
        for (int j = 0; j < s; ++j) {
            uint32_t y = Y[(long long)j * N + n];
            int i = 0;   // position of the first nonzero base-p digit of x = y / p^m
            if (y) {
                int t = 0;
                while (y >= (uint32_t)p) {
                    y /= (uint32_t)p;
                    ++t;
                }
                i = m - t;
            }
            kv *= 1.0 + gam[j] * kp[i];
            const double a = gam[j] * gam[j] * rp[i];
            rv *= 1.0 + a;
            out[(long long)(1 + j) * N + n] = rv;
            for (int q = j + 1; q >= 1; --q) e[q] += a * e[q - 1];
        }
        out[n] = kv;
        for (int q = 1; q <= s; ++q) out[(long long)(s + q) * N + n] = e[q];
    }
}

// real parts of the 1 + 2s transforms (interleaved complex when cplx) ->
// W_K = 1 / (N Re K~) and the tables, with R~_d(0) - 1
__global__ void k_spline_tables(const double* __restrict__ tr, int cplx, long long N, int s, double* W,
                                double* tab) {
    const long long total = (long long)(1 + 2 * s) * N;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total;
         x += (long long)gridDim.x * blockDim.x) {
        const long long row = x / N, H = x - row * N;
        const double v = cplx ? tr[2 * x] : tr[x];
        if (row == 0) {
            W[H] = 1.0 / ((double)N * v);
        } else {
            tab[x - N] = (row <= s && H == 0) ? v - 1.0 : v;
        }
    }
}

// c~ = f~ W_K in place ([batch][ld], real or interleaved complex): only where no
// variances are asked for (k_spline_dots scales on its way)
__global__ void k_spline_scale(double* ft, int cplx, long long N, long long ld, long long total,
                               const double* __restrict__ W) {
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total;
         x += (long long)gridDim.x * blockDim.x) {
        const long long b = x / N, H = x - b * N, o = b * ld + H;
        const double w = W[H];
        if (cplx) {
            ft[2 * o] *= w;
            ft[2 * o + 1] *= w;
        } else {
            ft[o] *= w;
        }
    }
}

// ---- the variance contraction ---------------------------------------------
// part[(b nt + t) ntile + tile] = sum over the tile's labels of |c~_b(H)|^2 T_t(H),
// and c~ = f~ W_K in place on the way.
//
// A batch of 32 functions against 32 tables is a matrix product with the labels
// as inner dimension, in FP64.  This GPU multiplies 1.7 FP64 numbers per clock
// and SM, so the product runs on the tensor cores in digits instead: in blocks
// of 64 labels every operand (for real data the square straight from c~'s
// significand, to 62 bits) becomes a 96-bit fixed-point number, scaled by its
// row's largest exponent so far in the tile, split into twelve signed digits of
// base 256 that FP16 holds exactly; a digit product is at most 2^14 and the
// 12 x 64 products that share a weight sum to less than 2^24, exact in FP32.
// The 78 digit pairs of weight >= 256^11 are multiplied; the sums join 128-bit
// integers per pair of function and table, in units of 2^88, shifted when a
// row's exponent grows.
//
// What is lost.  The products of digits are exact, the operands are not: fixed
// point has no exponent of its own, so a number keeps its 53 bits down to 2^-41
// of its row's largest and fewer below, and the digit pairs that are left out
// belong to the smaller numbers too.  Per label at most 2^95 for the two operands
// cut at one unit each (they stay below 2^94) and 11 2^14 2^80 (1 + 2^-7) for the
// pairs, together less than 2^10 units of the sum.  Where |c~|^2 is large the
// tables are small, so the largest product can lie far below the product of the
// largest; whether the bits kept were enough is therefore read off each result:
// a sum below 2^60 units per label, the error's bound then above 2^-50 of the sum,
// is formed again in FP64 by one warp.  (FP64 sums of 4096 labels, sixteen per
// thread and a tree over 256, are bound by 26 2^-53 > 2^-49.)  So are rows with an
// infinity, a NaN or a square near the largest number in the tile.  A pair's
// result depends on its own two rows only.
//
// Integer instructions and the tensor cores bound it, a fifth goes to the sums
// formed again.  p = 2, m = 20, s = 16, 32 functions: 2920 us on the FP64 pipe (one
// CTA per function and 4096 labels) plus 95 us for the scaling; so 608 us,
// 535 of them without the sums formed again (pair by pair instead of function by
// function 623; the next block's numbers loaded before this one's sums are drained,
// which takes 130 registers and spills, 708).  Eight digits, 36 pairs and no second look took
// 364 us and were wrong by up to 2^-16 of a variance (random values, s = 2, m = 16).
constexpr int kDotThreads = 256;
constexpr int kDotRows = 32;                  // functions, and tables, per round
constexpr int kDotK = 64;                     // labels per block
constexpr int kDotPlane = kDotRows * kDotK;   // halves of one digit's rows
constexpr int kDotDigits = 12;
constexpr int kDotOperand = kDotDigits * kDotPlane;   // halves of one operand
constexpr size_t kDotSmem = (size_t)2 * kDotOperand * 2 + 7 * kDotRows * 4 + 16;
constexpr int kDotKeep = 60;                  // log2 of the least sum per label that is kept

__device__ __forceinline__ uint32_t abs_hi(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// half of a digit plane: rows of 64 labels (128 bytes), their 16-byte pieces
// permuted by the row so that eight rows' same piece lies on all banks
__device__ __forceinline__ int plane_at(int row, int piece) { return row * kDotK + ((piece ^ (row & 7)) << 3); }

struct Fix96 {
    uint32_t w[3];   // low word first
};

// +-(v 2^32 2^-d) for v < 2^62, plus 128 in every byte with carries: byte - 128 is
// the signed digit; neg: all ones for minus (-v = ~v + 1)
__device__ __forceinline__ Fix96 place96(unsigned long long v, int d, uint32_t neg) {
    uint32_t a = 0, b = (uint32_t)v, c = (uint32_t)(v >> 32);
    d = min(d, 95);
    if (d >= 64) {
        a = c;
        b = c = 0;
    } else if (d >= 32) {
        a = b;
        b = c;
        c = 0;
    }
    const int r = d & 31;
    a = __funnelshift_r(a, b, r);
    b = __funnelshift_r(b, c, r);
    c >>= r;
    Fix96 x;
    asm("add.cc.u32 %0, %3, %6;\n addc.cc.u32 %1, %4, %7;\n addc.u32 %2, %5, %7;"
        : "=r"(x.w[0]), "=r"(x.w[1]), "=r"(x.w[2])
        : "r"(a ^ neg), "r"(b ^ neg), "r"(c ^ neg), "r"(0x80808080u - neg), "r"(0x80808080u));
    return x;
}

// x against exponent E (>= x's): significand 2^41 at E
template <bool SIGNED> __device__ __forceinline__ Fix96 to_fix96(double x, int E) {
    const uint32_t h = (uint32_t)__double2hiint(x);
    const int ex = (int)((h >> 20) & 0x7ffu);
    const uint32_t mh = (h & 0xfffffu) | (ex ? 0x100000u : 0u);
    const unsigned long long v = (((unsigned long long)mh << 32) | (uint32_t)__double2loint(x)) << 9;
    return place96(v, E - max(ex, 1), SIGNED ? (uint32_t)((int)h >> 31) : 0u);
}

// u^2 the same way, u's exponents against E: the top 62 of its 106 bits
__device__ __forceinline__ Fix96 square_fix96(double u, int E) {
    const uint32_t h = (uint32_t)__double2hiint(u), lo = (uint32_t)__double2loint(u);
    const int ex = (int)((h >> 20) & 0x7ffu);
    const uint32_t mh = (h & 0xfffffu) | (ex ? 0x100000u : 0u);
    const unsigned long long hh = (unsigned long long)mh * mh, mid = (unsigned long long)(2 * mh) * lo + __umulhi(lo, lo);
    return place96((hh << 20) + (mid >> 12), 2 * (E - max(ex, 1)), 0u);
}

// the digits of two numbers (label l and l + 32 of a block) into their planes
__device__ __forceinline__ void put_digits(__half* plane, int row, const Fix96& f0, const Fix96& f1, int lane) {
    const __half2 off = __halves2half2(__ushort_as_half(0xE480), __ushort_as_half(0xE480));   // -(1024 + 128)
    __half* p = plane + plane_at(row, lane >> 2) + 2 * (lane & 3);
#pragma unroll
    for (int i = 0; i < kDotDigits; ++i) {
        // bytes i of both behind 0x64: the FP16 numbers 1024 + byte
        const uint32_t sel = (uint32_t)(i & 3) | ((uint32_t)(4 + (i & 3)) << 4);
        const uint32_t two = __byte_perm(f0.w[i >> 2], f1.w[i >> 2], sel);
        const uint32_t bits = __byte_perm(two, 0x64u, 0x4140);
        __half2 h;
        memcpy(&h, &bits, 4);
        h = __hadd2(h, off);
        *reinterpret_cast<__half2*>(p + i * kDotPlane) = h;
    }
}

__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// sums over [h0, h1) of |c~|^2 T_t in FP64 by one warp, for the tables t of a mask:
// 256 labels at a time, their squares kept in registers for all tables; two chains
// per lane, then a tree.  Lane t returns table t's sum.
template <bool CPLX>
__device__ __forceinline__ double warp_sums(const double* c, const double* tab, long long N, unsigned mask, long long h0,
                                            long long h1, int lane) {
    double tot = 0.0;
    for (long long H = h0 + lane; H - lane < h1; H += 256) {
        double a[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const long long h = H + 32 * i;
            a[i] = 0.0;
            if (h >= h1) continue;
            if constexpr (CPLX) {
                const double2 u = reinterpret_cast<const double2*>(c)[h];
                a[i] = u.x * u.x + u.y * u.y;
            } else {
                a[i] = c[h] * c[h];
            }
        }
        for (unsigned m = mask; m; m &= m - 1) {
            const int tr = __ffs((int)m) - 1;
            const double* T = tab + (long long)tr * N;
            double y[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) y[i] = H + 32 * i < h1 ? T[H + 32 * i] : 0.0;
            double v0 = a[0] * y[0], v1 = a[1] * y[1];
#pragma unroll
            for (int i = 2; i < 8; i += 2) {
                v0 += a[i] * y[i];
                v1 += a[i + 1] * y[i + 1];
            }
            v0 += v1;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v0 += __shfl_xor_sync(0xffffffffu, v0, o);
            if (lane == tr) tot += v0;
        }
    }
    return tot;
}

// grid (tiles, groups of 32 functions); warp w converts rows 4 w .. 4 w + 3 of
// both operands and multiplies functions 16 (w & 1) .. + 15 by tables
// 8 (w >> 1) .. + 7
template <bool CPLX>
__global__ void __launch_bounds__(kDotThreads, 2) k_spline_dots(double* ct, long long N, long long ld, int batch, int nt,
                                                                const double* __restrict__ tab,
                                                                const double* __restrict__ W, double* part, int ntile,
                                                                int labels) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __half* A = reinterpret_cast<__half*>(smraw);
    __half* B = A + kDotOperand;
    int* grow = reinterpret_cast<int*>(B + kDotOperand);   // [2][32]: growth of the rows' exponents in this block
    int* bad = grow + 2 * kDotRows;                        // [2][32]: rows with an infinity or a NaN
    int* some = bad + 2 * kDotRows;                        // [2][32]: rows with a number other than zero
    unsigned* fails = reinterpret_cast<unsigned*>(some + 2 * kDotRows);   // [32]: a function's sums to form again
    int* next = reinterpret_cast<int*>(fails + kDotRows);
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int tile = blockIdx.x, f0 = blockIdx.y * kDotRows;
    const long long h0 = (long long)tile * labels, h1 = min(N, h0 + labels);
    const int fo = 16 * (w & 1), to = 8 * (w >> 1);
    // ldmatrix rows of this lane: A (16 rows x 16 labels of one digit), B (8 rows x 16
    // of two digits)
    const int ar = fo + (lane & 15), br = to + (lane & 7);
    const uint32_t arow = (uint32_t)__cvta_generic_to_shared(A + ar * kDotK);
    const uint32_t brow = (uint32_t)__cvta_generic_to_shared(B + (lane >> 4) * kDotPlane + br * kDotK);
    for (int t0 = 0; t0 < nt; t0 += kDotRows) {
        // top word of the first function-side number whose row takes FP64 sums: real
        // rows hold c~, whose square must not overflow
        constexpr int kDotPower = CPLX ? 1 : 2;   // powers of two of the sum per exponent of a function-side number
        constexpr uint32_t kDotHuge = CPLX ? 0x7ff00000u : (1023u + 511u) << 20;
        __syncthreads();
        if (t < 2 * kDotRows) bad[t] = 0;
        int Ea[4] = {1, 1, 1, 1}, Et[4] = {1, 1, 1, 1};   // exponents of this warp's rows
        unsigned any = 0;                                 // its rows with a number other than zero
        int ea[2] = {CPLX ? 1 : 2, CPLX ? 1 : 2}, et[2] = {1, 1};   // of the rows of this thread's sums
        long long hi[4] = {0, 0, 0, 0}, mid[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};   // sum = hi 2^64 + mid 2^32 + lo
        for (long long hb = h0; hb < h1; hb += kDotK) {
            const long long l0 = hb + lane, l1 = l0 + 32;
            const bool in0 = l0 < h1, in1 = l1 < h1;
            double a[4][2], x[4][2];
            {
                double w0 = 1.0, w1 = 1.0;
                if (t0 == 0 && in0) w0 = W[l0];
                if (t0 == 0 && in1) w1 = W[l1];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int f = f0 + 4 * w + k, tb = t0 + 4 * w + k;
                    a[k][0] = a[k][1] = x[k][0] = x[k][1] = 0.0;
                    if (f < batch) {
                        if constexpr (CPLX) {
                            double2* row = reinterpret_cast<double2*>(ct) + f * ld;
                            double2 u = in0 ? row[l0] : make_double2(0.0, 0.0), v = in1 ? row[l1] : make_double2(0.0, 0.0);
                            if (t0 == 0) {
                                u = make_double2(u.x * w0, u.y * w0);
                                v = make_double2(v.x * w1, v.y * w1);
                                if (in0) row[l0] = u;
                                if (in1) row[l1] = v;
                            }
                            a[k][0] = u.x * u.x + u.y * u.y;
                            a[k][1] = v.x * v.x + v.y * v.y;
                        } else {
                            double* row = ct + f * ld;
                            if (in0) a[k][0] = row[l0];
                            if (in1) a[k][1] = row[l1];
                        }
                    }
                    if (tb < nt) {
                        const double* row = tab + (long long)tb * N;
                        if (in0) x[k][0] = row[l0];
                        if (in1) x[k][1] = row[l1];
                    }
                }
                if constexpr (!CPLX) {
                    if (t0 == 0) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            a[k][0] *= w0;
                            a[k][1] *= w1;
                            if (f0 + 4 * w + k < batch) {
                                double* row = ct + (f0 + 4 * w + k) * ld;
                                if (in0) row[l0] = a[k][0];
                                if (in1) row[l1] = a[k][1];
                            }
                        }
                    }
                }
            }
            __syncthreads();   // the previous block's digits and growths have been read
            // the rows' largest exponents: eight reductions in flight
            uint32_t ma[4], mx[4], most = 0, least = 0xffffffffu;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                ma[k] = __reduce_max_sync(0xffffffffu, max(abs_hi(a[k][0]), abs_hi(a[k][1])));
                mx[k] = __reduce_max_sync(0xffffffffu, max(abs_hi(x[k][0]), abs_hi(x[k][1])));
                most = max(most, max(ma[k], mx[k]));
                least = min(least, min(ma[k], mx[k]));
            }
            if (least == 0) {   // a row of zeros, or of numbers whose top word is zero
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const double(&v)[2] = i < 4 ? a[i] : x[i - 4];
                    uint32_t& m = i < 4 ? ma[i] : mx[i - 4];
                    if (m == 0 && __any_sync(0xffffffffu, (__double2loint(v[0]) | __double2loint(v[1])) != 0)) m = 1;
                }
            }
            if (most >= kDotHuge) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    double(&v)[2] = i < 4 ? a[i] : x[i - 4];
                    uint32_t& m = i < 4 ? ma[i] : mx[i - 4];
                    if (m < (i < 4 ? kDotHuge : 0x7ff00000u)) continue;
                    bad[(i >> 2) * kDotRows + 4 * w + (i & 3)] = 1;
                    v[0] = v[1] = 0.0;
                    m = 0;
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int r = 4 * w + k;
                any |= (ma[k] ? 1u << k : 0u) | (mx[k] ? 16u << k : 0u);
                const int na = max((int)(ma[k] >> 20), Ea[k]), nx = max((int)(mx[k] >> 20), Et[k]);
                if (lane == 0) {
                    grow[r] = kDotPower * (na - Ea[k]);
                    grow[kDotRows + r] = nx - Et[k];
                }
                Ea[k] = na;
                Et[k] = nx;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int r = 4 * w + k;
                if constexpr (CPLX) put_digits(A, r, to_fix96<false>(a[k][0], Ea[k]), to_fix96<false>(a[k][1], Ea[k]), lane);
                else put_digits(A, r, square_fix96(a[k][0], Ea[k]), square_fix96(a[k][1], Ea[k]), lane);
                put_digits(B, r, to_fix96<true>(x[k][0], Et[k]), to_fix96<true>(x[k][1], Et[k]), lane);
            }
            __syncthreads();
            // the next block's lines on their way into L2: 64 rows of four
            if (const long long hn = hb + kDotK + 16 * (t & 3); hn < h1) {
                const int r = t >> 3;
                const double* p = t & 4 ? (t0 + r < nt ? tab + (long long)(t0 + r) * N + hn : nullptr)
                                        : (f0 + r < batch ? ct + ((f0 + r) * ld + hn) * (CPLX ? 2 : 1) : nullptr);
                if (p) asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
            }
            // weights 256^19 and up: at most 4 x 64 products of 2^14 onto 3 2^22, whose
            // last place is one: the sum is read off the bits
            float acc[kDotDigits][4];
#pragma unroll
            for (int c = 0; c < kDotDigits; ++c)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[c][q] = c < kDotDigits - 4 ? 0.f : 12582912.f;
#pragma unroll 1
            for (int k = 0; k < kDotK / 16; ++k) {
                const uint32_t aoff = arow + 16u * (uint32_t)((2 * k + (lane >> 4)) ^ (ar & 7));
                const uint32_t boff = brow + 16u * (uint32_t)((2 * k + ((lane >> 3) & 1)) ^ (br & 7));
                uint32_t fb[kDotDigits / 2][4];
#pragma unroll
                for (int j = 0; j < kDotDigits / 2; ++j) ldmatrix4(fb[j], boff + 2u * (uint32_t)(2 * j * kDotPlane));
#pragma unroll
                for (int i = 0; i < kDotDigits; ++i) {
                    uint32_t fa[4];
                    ldmatrix4(fa, aoff + 2u * (uint32_t)(i * kDotPlane));
#pragma unroll
                    for (int j = kDotDigits - 1 - i; j < kDotDigits; ++j)
                        mma_f16(acc[i + j - kDotDigits + 1], fa, fb[j >> 1][2 * (j & 1)], fb[j >> 1][2 * (j & 1) + 1]);
                }
            }
            // this thread's sums: rows fo + lane / 4 (+ 8), tables to + 2 (lane % 4) (+ 1)
            int ga[2], gt[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                ga[u] = grow[fo + (lane >> 2) + 8 * u];
                gt[u] = grow[kDotRows + to + 2 * (lane & 3) + u];
                ea[u] += ga[u];
                et[u] += gt[u];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int g = ga[q >> 1] + gt[q & 1];
                if (g) {
                    __int128 v = ((__int128)hi[q] << 64) + ((__int128)mid[q] << 32) + lo[q];
                    v = g > 126 ? (__int128)0 : v >> g;
                    hi[q] = (long long)(v >> 64);
                    mid[q] = (long long)((unsigned long long)(v >> 32) & 0xffffffffull);
                    lo[q] = (long long)((unsigned long long)v & 0xffffffffull);
                }
                auto whole = [&](int c) {
                    return c < kDotDigits - 4 ? __float2int_rn(acc[c][q]) : __float_as_int(acc[c][q]) - 0x4b400000;
                };
                // four weights: below 12 2^20 256^3 (1 + 2^-7) < 2^48
                auto four = [&](int c) {
                    return (long long)whole(c) + (long long)whole(c + 1) * 256 + (long long)whole(c + 2) * 65536 +
                           (long long)whole(c + 3) * 16777216;
                };
                lo[q] += four(0);
                mid[q] += four(4);
                hi[q] += four(8);
            }
        }
        if (lane < 8) some[(lane >> 2) * kDotRows + 4 * w + (lane & 3)] = (any >> lane) & 1;
        if (t < kDotRows) fails[t] = 0;
        if (t == 0) *next = 0;
        __syncthreads();   // bad and some are complete, c~ of the tile is written
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int fr = fo + (lane >> 2) + 8 * (q >> 1), tr = to + 2 * (lane & 3) + (q & 1);
            const int f = f0 + fr, tb = t0 + tr;
            if (f >= batch || tb >= nt) continue;
            const __int128 sum = ((__int128)hi[q] << 64) + ((__int128)mid[q] << 32) + lo[q];
            // digits of weight 256^11 and up; the unit of a row is 2^(E - 1116), of a
            // row of squares 2^(2 E - 2138)
            const long long top = (long long)(sum >> 60);   // below 2^52: nothing of weight is cut
            double v = scalbn((double)top * 0x1p60 + (double)(long long)((unsigned long long)sum & ((1ull << 60) - 1)),
                              88 + ea[q >> 1] + et[q & 1] - 1116 - (CPLX ? 1116 : 2138));
            bool redo = bad[fr] || bad[kDotRows + tr];
            if (!redo) {
                if (!some[fr] || !some[kDotRows + tr]) v = 0.0;
                else redo = sum < ((__int128)(h1 - h0) << kDotKeep);
            }
            if (redo) atomicOr(fails + fr, 1u << tr);
            else part[((long long)f * nt + tb) * ntile + tile] = v;
        }
        __syncthreads();
        for (;;) {   // the functions with sums to form again, one warp each
            int fr = 0;
            if (lane == 0) fr = atomicAdd(next, 1);
            fr = __shfl_sync(0xffffffffu, fr, 0);
            if (fr >= kDotRows) break;
            const unsigned mask = fails[fr];
            if (!mask) continue;
            const long long f = f0 + fr;
            const double v = warp_sums<CPLX>(ct + f * ld * (CPLX ? 2 : 1), tab + (long long)t0 * N, N, mask, h0, h1, lane);
            if ((mask >> lane) & 1) part[(f * nt + t0 + lane) * ntile + tile] = v;
        }
    }
}

// The same sums in FP64, for few functions or tables: a CTA scales one function's
// part of c~, keeps the squares in shared memory, and its warps take the tables in
// turn.  The FP64 pipe bounds it (an addition of a warp every 19 cycles per SM):
// p = 2, m = 20, one function, 4 / 32 / 128 tables: 20 / 91 / 329 us.
constexpr int kFewThreads = 256;
constexpr int kFewTile = 2048;   // labels per CTA at most

template <bool CPLX>
__global__ void __launch_bounds__(kFewThreads) k_spline_dots_fp64(double* ct, long long N, long long ld, int nt,
                                                                  const double* __restrict__ tab,
                                                                  const double* __restrict__ W, double* part, int ntile,
                                                                  int labels) {
    __shared__ double a[kFewTile];
    const long long b = blockIdx.y, h0 = (long long)blockIdx.x * labels;
    const int n = (int)min((long long)labels, N - h0), t = threadIdx.x, lane = t & 31;
    double* c = ct + b * ld * (CPLX ? 2 : 1);
    for (int i = t; i < n; i += kFewThreads) {
        const double w = W[h0 + i];
        if constexpr (CPLX) {
            double2* p = reinterpret_cast<double2*>(c) + h0 + i;
            const double2 u = make_double2(p->x * w, p->y * w);
            *p = u;
            a[i] = u.x * u.x + u.y * u.y;
        } else {
            const double u = c[h0 + i] * w;
            c[h0 + i] = u;
            a[i] = u * u;
        }
    }
    __syncthreads();
    for (int tb = t >> 5; tb < nt; tb += kFewThreads / 32) {
        const double* T = tab + (long long)tb * N + h0;
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        for (int i0 = lane; i0 < n; i0 += 256) {   // eight loads in flight
            double x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = i0 + 32 * k < n ? T[i0 + 32 * k] : 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (i0 + 32 * k < n) v[k & 3] += a[i0 + 32 * k] * x[k];
        }
        double x = (v[0] + v[1]) + (v[2] + v[3]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) part[(b * nt + tb) * ntile + blockIdx.x] = x;
    }
}

// sums over tiles, then the cumulative variances and dimensions (least d with
// variance >= thr * total, 0 when the total is 0): one CTA per function, or a
// cluster whose sums meet in the first CTA's shared memory.  The FP64 additions of
// the 2 s ntile partials bound it (p = 2, m = 20, s = 16, 32 functions, 4096 tiles:
// 48 us with one CTA, 23 us in a cluster of eight).
constexpr int kFinThreads = 512;
template <int CL>
__global__ void __launch_bounds__(kFinThreads) k_spline_finalize(const double* __restrict__ part, int ntile, int s,
                                                                 int lg, double N2, double thr, double* var_trc,
                                                                 double* var_sup, int* dim) {
    namespace cg = cooperative_groups;
    __shared__ double x[2 * kSplineMaxS];
    __shared__ double v[2][kSplineMaxS + 1];
    __shared__ int first[2];
    const long long b = blockIdx.x / CL;
    const int t = threadIdx.x, rank = blockIdx.x % CL;
    double* dst = x;
    if constexpr (CL > 1) {
        dst = cg::this_cluster().map_shared_rank(x, 0);
        cg::this_cluster().sync();   // the first CTA is running before its shared memory is written
    }
    sum_rows(part + b * 2 * s * ntile, 2 * s, ntile, lg, rank, CL, dst);
    if constexpr (CL > 1) {
        cg::this_cluster().sync();
        if (rank != 0) return;
    }
    if (t < 2) first[t] = s;
    __syncthreads();
    if (t == 0) {
        double acc = v[1][0] = 0.0;
        for (int d = 1; d <= s; ++d) v[1][d] = acc += N2 * x[s + d - 1];
    } else if (t >= 32 && t <= 32 + s) {
        v[0][t - 32] = t == 32 ? 0.0 : N2 * x[t - 33];
    }
    __syncthreads();
    if (t <= s) {
        if (var_trc) var_trc[b * (s + 1) + t] = v[0][t];
        if (var_sup) var_sup[b * (s + 1) + t] = v[1][t];
        const double lim = thr * v[0][s];
        if (v[0][t] >= lim) atomicMin(first, t);
        if (v[1][t] >= lim) atomicMin(first + 1, t);
    }
    __syncthreads();
    if (t < 2 && dim) dim[2 * b + t] = v[0][s] > 0.0 ? first[t] : 0;
}

// kernel data at the shifted points: Kd[w] = prod_j (1 + gamma_j K'(x_{j,w} (+) delta_j, 0)),
// x_{j,w} with m digits, delta_j = D[j] / p^M with M digits; kpM[i] = K' for a first
// nonzero digit at position i of M (kpM[0] = 1)
__global__ void k_spline_shift_data(const uint32_t* __restrict__ Y, long long N, int s, int p, int m, int M,
                                    const uint32_t* __restrict__ D, const double* __restrict__ kpM,
                                    const double* __restrict__ gam, double* Kd) {
    unsigned long long up = 1;
    for (int i = m; i < M; ++i) up *= (unsigned long long)p;
    for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < N; w += (long long)gridDim.x * blockDim.x) {
        double kv = 1.0;
        for (int j = 0; j < s; ++j) {
            unsigned long long a = (unsigned long long)Y[(long long)j * N + w] * up, b = D[j], y;
            if (p == 2) {
                y = a ^ b;
            } else {
                y = 0;
                unsigned long long pw = 1;
                for (int c = 0; c < M; ++c) {
                    y += ((a % p + b % p) % p) * pw;
                    a /= p;
                    b /= p;
                    pw *= p;
                }
            }
            int i = 0;
            if (y) {
                int t = 0;
                while (y >= (unsigned long long)p) {
                    y /= p;
                    ++t;
                }
                i = M - t;
            }
            kv *= 1.0 + gam[j] * kpM[i];
        }
        Kd[w] = kv;
    }
}

// g~ = N c~ k~ in place in c~ (real, or interleaved complex with k~ complex)
__global__ void k_spline_conv(double* ct, const double* __restrict__ kt, int cplx, long long N, long long total) {
    const double n = (double)N;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total;
         x += (long long)gridDim.x * blockDim.x) {
        const long long H = x % N;
        if (cplx) {
            const double ar = ct[2 * x], ai = ct[2 * x + 1], br = kt[2 * H], bi = kt[2 * H + 1];
            ct[2 * x] = n * (ar * br - ai * bi);
            ct[2 * x + 1] = n * (ar * bi + ai * br);
        } else {
            ct[x] *= n * kt[H];
        }
    }
}

// per-block partial sums of (f - Re v)^2 over a tile of points; part[b * ntile + tile]
__global__ void __launch_bounds__(256) k_spline_sse(const double* __restrict__ f, const double* __restrict__ v,
                                                    int cplx, long long N, long long ld, double* part,
                                                    long long ntile) {
    __shared__ double red[256];
    const long long tile = blockIdx.x, b = blockIdx.y;
    double acc = 0.0;
    for (int q = 0; q < kDotTile / 256; ++q) {
        const long long n = tile * kDotTile + threadIdx.x + 256 * q;
        if (n < N) {
            const long long x = b * ld + n;
            const double d = f[x] - (cplx ? v[2 * x] : v[x]);
            acc += d * d;
        }
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[b * ntile + tile] = red[0];
}

__global__ void k_spline_sse_final(const double* __restrict__ part, long long ntile, int batch, double* sse) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= batch) return;
    double x = 0.0;
    for (long long i = 0; i < ntile; ++i) x += part[(long long)b * ntile + i];
    sse[b] = x;
}

// ---- the spline at arbitrary points (Sec. 3.1) ----------------------------
// K(x (-) x_n, 0) = prod_j (1 + gamma_j K'(x_j (-) x_{j,n}, 0)), and K' depends
// only on the position i of the first nonzero digit of the difference: the
// first digit (of m) where x_j and the net point differ, or, when the top m
// digits agree, the first nonzero digit of x_j below them (0 if none).  With
// the base-p digits packed BP bits each (1, 2, 3, 4, 5 bits for p = 2, 3, 5 / 7,
// 11 / 13, 17 .. 31), the first differing digit is the highest set bit of an XOR.
constexpr int kEvalQB = 128;   // points per block, one per thread
constexpr int kEvalFB = 8;     // functions per block

__host__ __device__ inline int eval_bits(int p) { return p == 2 ? 1 : p == 3 ? 2 : p <= 7 ? 3 : p <= 15 ? 4 : 5; }

__device__ __forceinline__ unsigned long long pack_digits(uint32_t v, int p, int m, int bp) {
    unsigned long long r = 0;
    for (int k = 0; k < m; ++k) {
        r |= (unsigned long long)(v % (uint32_t)p) << (bp * k);
        v /= (uint32_t)p;
    }
    return r;
}

// packed top-m digits of the net points, [s][N]
__global__ void k_eval_pack(const uint32_t* __restrict__ Y, long long total, int p, int m,
                            unsigned long long* __restrict__ PY) {
    const int bp = eval_bits(p);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x)
        PY[e] = p == 2 ? (unsigned long long)Y[e] : pack_digits(Y[e], p, m, bp);
}

// Partial sums over one chunk of the net (blockIdx.z) for kEvalQB points
// (blockIdx.x) and kEvalFB functions (blockIdx.y):
//   part[z][f][q] = sum_{n in chunk} Re c[f][n] prod_j T[j][i_j(q, n)],
// T[j][i] = 1 + gamma_j K'(i) (i = 0 .. M).  The net points and coefficients
// of the chunk pass through shared memory in tiles of TN; each thread keeps
// its point's packed digits and tail positions in shared memory too.
template <int P>
__global__ void __launch_bounds__(kEvalQB) k_spline_eval(const unsigned long long* __restrict__ PY, long long N,
                                                          const double* __restrict__ c, long long ldc, int cstride,
                                                          int batch, const uint32_t* __restrict__ X, int Q, int s,
                                                          int m, int M, const double* __restrict__ Tg,
                                                          long long chunk, int TN, double* __restrict__ part) {
    constexpr int p = P;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int M1 = M + 1;
    double* T = reinterpret_cast<double*>(smraw);                                   // [s][M+1]
    unsigned long long* PX = reinterpret_cast<unsigned long long*>(T + (size_t)s * M1);   // [s][QB]
    unsigned long long* PYs = PX + (size_t)s * kEvalQB;                             // [s][TN]
    double* cs = reinterpret_cast<double*>(PYs + (size_t)s * TN);                   // [FB][TN]
    unsigned char* tl = reinterpret_cast<unsigned char*>(cs + (size_t)kEvalFB * TN);   // [s][QB]
    const int t = threadIdx.x;
    const int q = blockIdx.x * kEvalQB + t;
    const int f0 = blockIdx.y * kEvalFB;
    const int nf = min(kEvalFB, batch - f0);
    constexpr int bp = P == 2 ? 1 : P == 3 ? 2 : P <= 7 ? 3 : P <= 15 ? 4 : 5;   // eval_bits(P)
    for (int e = t; e < s * M1; e += blockDim.x) T[e] = Tg[e];
    {
        uint32_t up = 1;
        for (int k = 0; k < M - m; ++k) up *= (uint32_t)p;
        for (int j = 0; j < s; ++j) {
            const uint32_t x = q < Q ? X[(long long)q * s + j] : 0u;
            const uint32_t top = up > 1 ? x / up : x, tail = up > 1 ? x % up : 0u;
            PX[j * kEvalQB + t] = p == 2 ? (unsigned long long)top : pack_digits(top, p, m, bp);
            int tp = 0;   // first nonzero digit of the tail, as a position in 1..M
            if (tail) {
                int e = 0;
                for (uint32_t v = tail; v >= (uint32_t)p; v /= (uint32_t)p) ++e;
                tp = M - e;
            }
            tl[j * kEvalQB + t] = (unsigned char)tp;
        }
    }
    double acc[kEvalFB];
#pragma unroll
    for (int f = 0; f < kEvalFB; ++f) acc[f] = 0.0;
    const long long n0 = blockIdx.z * chunk, n1 = min(N, n0 + chunk);
    for (long long nb = n0; nb < n1; nb += TN) {
        const int tn = (int)min((long long)TN, n1 - nb);
        __syncthreads();   // the previous tile is consumed (and the tables above are written)
        for (int e = t; e < s * TN; e += blockDim.x) {
            const int j = e / TN, u = e - j * TN;
            PYs[e] = u < tn ? PY[(long long)j * N + nb + u] : 0ull;
        }
        for (int e = t; e < kEvalFB * TN; e += blockDim.x) {
            const int f = e / TN, u = e - f * TN;
            cs[e] = (f < nf && u < tn) ? c[(long long)(f0 + f) * ldc + (nb + u) * cstride] : 0.0;
        }
        __syncthreads();
        for (int u = 0; u < tn; ++u) {
            // two partial products (even and odd coordinates) keep two
            // multiplication chains in flight
            double pr0 = 1.0, pr1 = 1.0;
            int j = 0;
            for (; j + 1 < s; j += 2) {
                const unsigned long long d0 = PX[j * kEvalQB + t] ^ PYs[j * TN + u];
                const unsigned long long d1 = PX[(j + 1) * kEvalQB + t] ^ PYs[(j + 1) * TN + u];
                const int i0 = d0 ? m - (63 - __clzll((long long)d0)) / bp : (int)tl[j * kEvalQB + t];
                const int i1 = d1 ? m - (63 - __clzll((long long)d1)) / bp : (int)tl[(j + 1) * kEvalQB + t];
                pr0 *= T[j * M1 + i0];
                pr1 *= T[(j + 1) * M1 + i1];
            }
            if (j < s) {
                const unsigned long long d0 = PX[j * kEvalQB + t] ^ PYs[j * TN + u];
                const int i0 = d0 ? m - (63 - __clzll((long long)d0)) / bp : (int)tl[j * kEvalQB + t];
                pr0 *= T[j * M1 + i0];
            }
            const double prod = pr0 * pr1;
#pragma unroll
            for (int f = 0; f < kEvalFB; ++f) acc[f] = fma(cs[f * TN + u], prod, acc[f]);
        }
    }
    if (q < Q) {
        for (int f = 0; f < nf; ++f) part[((long long)blockIdx.z * batch + f0 + f) * Q + q] = acc[f];
    }
}

// values[f][q] = sum over the chunks in order
__global__ void k_spline_eval_reduce(const double* __restrict__ part, int nch, int batch, int Q,
                                     double* __restrict__ values, long long ldv) {
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e >= (long long)batch * Q) return;
    const long long f = e / Q, q = e - f * Q;
    double a = 0.0;
    for (int z = 0; z < nch; ++z) a += part[(long long)z * batch * Q + e];
    values[f * ldv + q] = a;
}

unsigned grid_sp(long long n) { return (unsigned)std::max(1ll, std::min((n + 255) / 256, 8ll * 152)); }

}  // namespace

void spline_free(dwt_plan_s* P, cudaStream_t st, bool sync) {
    if (sync) {
        cudaFree(P->d_splW);
        cudaFree(P->d_splT);
    } else {
        dfree(P->d_splW, st);
        dfree(P->d_splT, st);
    }
    P->d_splW = nullptr;
    P->d_splT = nullptr;
}

int run_spline_prepare(dwt_plan_s* P, double alpha, const double* gamma, cudaStream_t st) {
    const long long N = P->N;
    const int s = P->s, p = P->p, m = P->m;
    if (s > kSplineMaxS) {
        set_error("the kernel spline supports s <= %d", kSplineMaxS);
        return DWT_EUNSUPPORTED;
    }
    // K'(x, 0) and R'(x, 0) by the position i (1..m) of the first nonzero digit; i = 0 for x = 0
    std::vector<double> hv(3 * (m + 1) + s);
    const double pa = std::pow((double)p, alpha), p2a = std::pow((double)p, 2.0 * alpha);
    const double rc = (pa - p) * (pa - p) / ((p - 1.0) * (p2a - p));
    for (int i = 0; i <= m; ++i) {
        hv[i] = i == 0 ? 1.0 : 1.0 - std::pow((double)p, i * (1.0 - alpha)) * (pa - 1.0) / (p - 1.0);
        hv[m + 1 + i] = i == 0 ? rc : rc * (1.0 - std::pow((double)p, i * (1.0 - 2.0 * alpha)) * (p2a - 1.0) / (p - 1.0));
    }
    for (int j = 0; j < s; ++j) hv[2 * (m + 1) + j] = gamma[j];
    const int rows = 1 + 2 * s;
    const bool cplx = p != 2;
    uint32_t* Y = nullptr;
    double *dv = nullptr, *data = nullptr, *tr = nullptr;
    auto cleanup = [&]() {
        dfree(Y, st);
        dfree(dv, st);
        dfree(data, st);
        if (tr != data) dfree(tr, st);
    };
    if (dmalloc((void**)&Y, (size_t)s * N * 4, st) || dmalloc((void**)&dv, hv.size() * 8, st) ||
        dmalloc((void**)&data, (size_t)rows * N * 8, st)) {
        cleanup();
        return DWT_ENOMEM;
    }
    tr = data;
    if (cplx && dmalloc((void**)&tr, (size_t)rows * N * 16, st)) {
        tr = data;
        cleanup();
        return DWT_ENOMEM;
    }
    DWT_CK(cudaMemcpyAsync(dv, hv.data(), hv.size() * 8, cudaMemcpyHostToDevice, st));
    int rc2 = run_points(P, Y, N, st);
    if (rc2) { cleanup(); return rc2; }
    {
        LaunchScope ls("spline_data", st);
        k_spline_data<<<grid_sp(N), 128, 0, st>>>(Y, N, s, p, m, dv, dv + m + 1, dv + 2 * (m + 1), data);
    }
    DWT_CK_LAUNCH("k_spline_data");
    rc2 = run_transform(P, data, tr, rows, N, N, DWT_F64, cplx ? DWT_C128 : DWT_F64, -1, st);
    if (rc2) { cleanup(); return rc2; }
    spline_free(P, st, false);
    P->spl_alpha = alpha;
    P->spl_gamma.assign(gamma, gamma + s);
    if (dmalloc((void**)&P->d_splW, (size_t)N * 8, st) || dmalloc((void**)&P->d_splT, (size_t)2 * s * N * 8, st)) {
        spline_free(P, st, false);
        cleanup();
        return DWT_ENOMEM;
    }
    {
        LaunchScope ls("spline_tables", st);
        k_spline_tables<<<grid_sp((long long)rows * N), 256, 0, st>>>(tr, cplx ? 1 : 0, N, s, P->d_splW, P->d_splT);
    }
    DWT_CK_LAUNCH("k_spline_tables");
    cleanup();
    return DWT_OK;
}

int run_spline_shifted(dwt_plan_s* P, const void* c, const uint32_t* delta, int M, void* values, int batch,
                       long long ld, const double* f_shift, double* sse, cudaStream_t st) {
    if (!P->d_splW) {
        set_error("dwt_spline_values_shifted: no kernel tables (call dwt_spline_prepare first)");
        return DWT_EINVAL;
    }
    const long long N = P->N;
    const int s = P->s, p = P->p, m = P->m;
    if (M < m || (double)M * std::log2((double)p) > 32.0) {
        set_error("dwt_spline_values_shifted: need m <= M and p^M <= 2^32");
        return DWT_EINVAL;
    }
    const bool cplx = p != 2;
    const size_t eb = cplx ? 16 : 8;
    // K'(y, 0) on M digits by the first nonzero digit, and the kernel weights
    const double alpha = P->spl_alpha;
    const double pa = std::pow((double)p, alpha);
    std::vector<double> hv((size_t)M + 1 + s);
    for (int i = 0; i <= M; ++i)
        hv[i] = i == 0 ? 1.0 : 1.0 - std::pow((double)p, i * (1.0 - alpha)) * (pa - 1.0) / (p - 1.0);
    for (int j = 0; j < s; ++j) hv[M + 1 + j] = P->spl_gamma[j];
    uint32_t *Y = nullptr, *dD = nullptr;
    double *dv = nullptr, *kd = nullptr, *kt = nullptr, *ct = nullptr, *part = nullptr;
    auto cleanup = [&]() {
        dfree(Y, st); dfree(dD, st); dfree(dv, st); dfree(kd, st); dfree(kt, st); dfree(ct, st); dfree(part, st);
    };
    const long long ntile = (N + kDotTile - 1) / kDotTile;
    if (dmalloc((void**)&Y, (size_t)s * N * 4, st) || dmalloc((void**)&dD, (size_t)s * 4, st) ||
        dmalloc((void**)&dv, hv.size() * 8, st) || dmalloc((void**)&kd, (size_t)N * 8, st) ||
        dmalloc((void**)&kt, (size_t)N * eb, st) || dmalloc((void**)&ct, (size_t)batch * N * eb, st) ||
        (sse && f_shift && dmalloc((void**)&part, (size_t)batch * ntile * 8, st))) {
        cleanup();
        return DWT_ENOMEM;
    }
    DWT_CK(cudaMemcpyAsync(dv, hv.data(), hv.size() * 8, cudaMemcpyHostToDevice, st));
    DWT_CK(cudaMemcpyAsync(dD, delta, (size_t)s * 4, cudaMemcpyHostToDevice, st));
    int rc = run_points(P, Y, N, st);
    if (rc) { cleanup(); return rc; }
    {
        LaunchScope ls("spline_shift_data", st);
        k_spline_shift_data<<<grid_sp(N), 128, 0, st>>>(Y, N, s, p, m, M, dD, dv, dv + M + 1, kd);
    }
    DWT_CK_LAUNCH("k_spline_shift_data");
    const dwt_dtype ct_t = cplx ? DWT_C128 : DWT_F64;
    if ((rc = run_transform(P, kd, kt, 1, N, N, DWT_F64, ct_t, -1, st)) ||
        (rc = run_transform(P, c, ct, batch, ld, N, ct_t, ct_t, -1, st))) {
        cleanup();
        return rc;
    }
    {
        LaunchScope ls("spline_conv", st);
        k_spline_conv<<<grid_sp((long long)batch * N), 256, 0, st>>>(ct, kt, cplx ? 1 : 0, N, (long long)batch * N);
    }
    DWT_CK_LAUNCH("k_spline_conv");
    if ((rc = run_transform(P, ct, values, batch, N, ld, ct_t, ct_t, +1, st))) {
        cleanup();
        return rc;
    }
    if (sse && f_shift) {
        for (int b0 = 0; b0 < batch; b0 += 65535) {
            const int nb = std::min(65535, batch - b0);
            LaunchScope ls("spline_sse", st);
            k_spline_sse<<<dim3((unsigned)ntile, (unsigned)nb), 256, 0, st>>>(
                f_shift + (size_t)b0 * ld, reinterpret_cast<const double*>(values) + (size_t)b0 * ld * (eb / 8),
                cplx ? 1 : 0, N, ld, part + (size_t)b0 * ntile, ntile);
        }
        LaunchScope ls("spline_sse", st);
        k_spline_sse_final<<<(batch + 127) / 128, 128, 0, st>>>(part, ntile, batch, sse);
    }
    DWT_CK_LAUNCH("k_spline_sse");
    cleanup();
    return DWT_OK;
}

int run_spline_eval(dwt_plan_s* P, const void* c, int batch, long long ld, const uint32_t* X, int Q, int M,
                    double* values, long long ldv, cudaStream_t st) {
    if (!P->d_splW) {
        set_error("dwt_spline_eval: no kernel (call dwt_spline_prepare first)");
        return DWT_EINVAL;
    }
    const long long N = P->N;
    const int s = P->s, p = P->p, m = P->m;
    if (M < m || (double)M * std::log2((double)p) > 32.0) {
        set_error("dwt_spline_eval: need m <= M and p^M <= 2^32");
        return DWT_EINVAL;
    }
    if (Q == 0) return DWT_OK;
    // T[j][i] = 1 + gamma_j K'(i) on M digits
    const double alpha = P->spl_alpha;
    const double pa = std::pow((double)p, alpha);
    std::vector<double> hT((size_t)s * (M + 1));
    for (int j = 0; j < s; ++j)
        for (int i = 0; i <= M; ++i) {
            const double kp = i == 0 ? 1.0 : 1.0 - std::pow((double)p, i * (1.0 - alpha)) * (pa - 1.0) / (p - 1.0);
            hT[(size_t)j * (M + 1) + i] = 1.0 + P->spl_gamma[j] * kp;
        }
    // tiles of the net: TN points, within the shared-memory budget
    const int TN = s > 32 ? 64 : 128;
    const size_t smem = (size_t)s * (M + 1) * 8 + (size_t)s * kEvalQB * 8 + (size_t)s * TN * 8 +
                        (size_t)kEvalFB * TN * 8 + (size_t)s * kEvalQB;
    int dev = 0, sms = 0;
    DWT_CK(cudaGetDevice(&dev));
    DWT_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int qb = (Q + kEvalQB - 1) / kEvalQB, fb = (batch + kEvalFB - 1) / kEvalFB;
    const long long ntn = (N + TN - 1) / TN;
    long long nch = std::max(1ll, std::min(ntn, (4ll * sms + (long long)qb * fb - 1) / ((long long)qb * fb)));
    nch = std::min(nch, 65535ll);
    const long long chunk = (ntn + nch - 1) / nch * TN;
    nch = (N + chunk - 1) / chunk;
    if (fb > 65535 || qb > (1 << 30)) {
        set_error("dwt_spline_eval: too many functions in one call");
        return DWT_EINVAL;
    }
    uint32_t* Y = nullptr;
    unsigned long long* PY = nullptr;
    double *dT = nullptr, *part = nullptr;
    auto cleanup = [&]() { dfree(Y, st); dfree(PY, st); dfree(dT, st); dfree(part, st); };
    if (dmalloc((void**)&Y, (size_t)s * N * 4, st) || dmalloc((void**)&PY, (size_t)s * N * 8, st) ||
        dmalloc((void**)&dT, hT.size() * 8, st) || dmalloc((void**)&part, (size_t)nch * batch * Q * 8, st)) {
        cleanup();
        return DWT_ENOMEM;
    }
    DWT_CK(cudaMemcpyAsync(dT, hT.data(), hT.size() * 8, cudaMemcpyHostToDevice, st));
    int rc = run_points(P, Y, N, st);
    if (rc) { cleanup(); return rc; }
    {
        LaunchScope ls("spline_eval_pack", st);
        k_eval_pack<<<grid_sp((long long)s * N), 256, 0, st>>>(Y, (long long)s * N, p, m, PY);
    }
    DWT_CK_LAUNCH("k_eval_pack");
    {
        auto kern = k_spline_eval<2>;
        switch (p) {
            case 3: kern = k_spline_eval<3>; break;
            case 5: kern = k_spline_eval<5>; break;
            case 7: kern = k_spline_eval<7>; break;
            case 11: kern = k_spline_eval<11>; break;
            case 13: kern = k_spline_eval<13>; break;
            case 17: kern = k_spline_eval<17>; break;
            case 19: kern = k_spline_eval<19>; break;
            case 23: kern = k_spline_eval<23>; break;
            case 29: kern = k_spline_eval<29>; break;
            case 31: kern = k_spline_eval<31>; break;
            default: break;
        }
        if ((rc = smem_limit_max(kern))) { cleanup(); return rc; }
        LaunchScope ls("spline_eval", st);
        kern<<<dim3((unsigned)qb, (unsigned)fb, (unsigned)nch), kEvalQB, smem, st>>>(
            PY, N, reinterpret_cast<const double*>(c), (p == 2 ? 1 : 2) * ld, p == 2 ? 1 : 2, batch, X, Q, s, m, M,
            dT, chunk, TN, part);
    }
    DWT_CK_LAUNCH("k_spline_eval");
    {
        LaunchScope ls("spline_eval_reduce", st);
        const long long tot = (long long)batch * Q;
        k_spline_eval_reduce<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(part, (int)nch, batch, Q, values, ldv);
    }
    DWT_CK_LAUNCH("k_spline_eval_reduce");
    cleanup();
    return DWT_OK;
}

template <int CL>
static int launch_finalize_cl(const double* part, int nb, int ntile, int s, double N2, double thr, double* vt, double* vs,
                              int* dim, cudaStream_t st) {
    LaunchScope ls("spline_finalize", st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nb * CL);
    cfg.blockDim = dim3(kFinThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {CL, 1, 1};
    cfg.attrs = at;
    cfg.numAttrs = CL > 1 ? 1 : 0;
    const int lg = sum_rows_lanes((2 * s + CL - 1) / CL, ntile, kFinThreads);
    DWT_CK(cudaLaunchKernelEx(&cfg, k_spline_finalize<CL>, part, ntile, s, lg, N2, thr, vt, vs, dim));
    return DWT_OK;
}
// a cluster from 2049 partials per function, as in effdim_reduce
static int launch_finalize(const double* part, int nb, int ntile, int s, double N2, double thr, double* vt, double* vs,
                           int* dim, cudaStream_t st) {
    return 2ll * s * ntile <= 2048 ? launch_finalize_cl<1>(part, nb, ntile, s, N2, thr, vt, vs, dim, st)
                                   : launch_finalize_cl<8>(part, nb, ntile, s, N2, thr, vt, vs, dim, st);
}

int run_spline(dwt_plan_s* P, const double* f, void* c, int batch, long long ld, double* var_trc, double* var_sup,
               int* dim, double thr, cudaStream_t st) {
    if (!P->d_splW) {
        set_error("dwt_spline: no kernel tables (call dwt_spline_prepare first)");
        return DWT_EINVAL;
    }
    const long long N = P->N;
    const int s = P->s;
    const bool cplx = P->p != 2;
    const size_t eb = cplx ? 16 : 8;
    // f~ and c~ lie in c when there is one (the transforms run in place), unless
    // it shares memory with f in another way than p = 2's in place
    const size_t rows = (size_t)(batch - 1) * ld + N;
    const char *f0 = reinterpret_cast<const char*>(f), *c0 = reinterpret_cast<const char*>(c);
    const bool apart = f0 + rows * 8 <= c0 || c0 + rows * eb <= f0;
    const bool own = !c || !(apart || (!cplx && f0 == c0));
    double* ft = reinterpret_cast<double*>(c);
    const long long ldt = own ? N : ld;
    double* part = nullptr;
    const bool want_var = var_trc || var_sup || dim;
    const long long groups = ((long long)batch + kDotRows - 1) / kDotRows, rounds = (2 * s + kDotRows - 1) / kDotRows;
    // a round of up to 32 functions and 32 tables costs as much in digits as 300 pairs
    // in FP64 (2^20 points, contraction: 9 x 32 pairs 621 us in FP64, 10 x 32 591 us in
    // digits; 30 x 10 722, 32 x 10 676; 2^16 points 79 and 54 us; 3^12 344 and 406);
    // with fewer the FP64 form is faster (1 x 4 pairs 20 us, 361 us before in digits)
    const bool few = (long long)batch * 2 * s <= 300 * groups * rounds;
    // labels per tile, from the net alone: a function's sums do not depend on the
    // others of its call.  Tiles for two CTAs per SM of one group; in digits at most
    // 256 labels (the sums that are formed again in FP64 find the tile in L2, fewer
    // fail and no SM is left with a long list: p = 2, 32 functions of s = 16, pair by
    // pair, contraction of smooth functions, 2048 / 1024 / 512 / 256 labels: m = 20
    // 880 / 744 / 651 / 623 us, m = 18 - / 286 / 221 / 174, random values 1418 / 878 /
    // 707 / 638 and - / 509 / 368 / 267) or 16 s, so that the tiles' sums take a byte
    // per point at most; in FP64 between 256 and 2048
    long long labels = (N + P->min_tiles - 1) / P->min_tiles;
    if (few) labels = std::min<long long>(kFewTile, std::max(256ll, (labels + 255) / 256 * 256));
    else labels = std::min<long long>(std::max(256, s / 4 * kDotK), (labels + kDotK - 1) / kDotK * kDotK);
    const int ntile = (int)((N + labels - 1) / labels);
    // functions per launch: the tiles' sums within 512 MB, one group of 32 at least
    const long long most = std::max(1ll, (64ll << 20) / ((long long)2 * s * ntile * kDotRows)) * kDotRows;
    const int chunk = (int)std::min<long long>(batch, std::min(most, few ? 65504ll : 65535ll * kDotRows));
    if ((own && dmalloc((void**)&ft, (size_t)batch * N * eb, st)) ||
        (want_var && dmalloc((void**)&part, (size_t)chunk * 2 * s * ntile * 8, st))) {
        if (own) dfree(ft, st);
        return DWT_ENOMEM;
    }
    auto cleanup = [&]() {
        if (own) dfree(ft, st);
        dfree(part, st);
    };
    int rc = run_transform(P, f, ft, batch, ld, ldt, DWT_F64, cplx ? DWT_C128 : DWT_F64, -1, st);
    if (rc) { cleanup(); return rc; }
    if (want_var) {
        auto kern = cplx ? k_spline_dots<true> : k_spline_dots<false>;
        auto kern64 = cplx ? k_spline_dots_fp64<true> : k_spline_dots_fp64<false>;
        if ((rc = smem_limit_max(kern))) { cleanup(); return rc; }
        for (long long b0 = 0; b0 < batch; b0 += chunk) {
            const int nb = (int)std::min<long long>(chunk, batch - b0);
            double* rows0 = ft + b0 * ldt * (cplx ? 2 : 1);
            if (few) {
                LaunchScope ls("spline_dots_fp64", st);
                kern64<<<dim3((unsigned)ntile, (unsigned)nb), kFewThreads, 0, st>>>(rows0, N, ldt, 2 * s, P->d_splT,
                                                                                    P->d_splW, part, ntile, (int)labels);
            } else {
                LaunchScope ls("spline_dots", st);
                kern<<<dim3((unsigned)ntile, (unsigned)((nb + kDotRows - 1) / kDotRows)), kDotThreads, kDotSmem, st>>>(
                    rows0, N, ldt, nb, 2 * s, P->d_splT, P->d_splW, part, ntile, (int)labels);
            }
            DWT_CK_LAUNCH("k_spline_dots");
            double* vt = var_trc ? var_trc + b0 * (s + 1) : nullptr;
            double* vs = var_sup ? var_sup + b0 * (s + 1) : nullptr;
            rc = launch_finalize(part, nb, ntile, s, (double)N * (double)N, thr, vt, vs, dim ? dim + 2 * b0 : nullptr, st);
            if (rc) { cleanup(); return rc; }
        }
    } else {
        LaunchScope ls("spline_scale", st);
        k_spline_scale<<<grid_sp((long long)batch * N), 256, 0, st>>>(ft, cplx ? 1 : 0, N, ldt, (long long)batch * N,
                                                                     P->d_splW);
    }
    DWT_CK_LAUNCH("k_spline_scale");
    if (c) {
        rc = run_transform(P, ft, c, batch, ldt, ld, cplx ? DWT_C128 : DWT_F64, cplx ? DWT_C128 : DWT_F64, +1, st);
        if (rc) { cleanup(); return rc; }
    }
    cleanup();
    return DWT_OK;
}

}  // namespace dwt
