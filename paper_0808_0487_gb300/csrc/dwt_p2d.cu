// dwt_p2d.cu -- the p = 2 transform in FP64 (Algorithms 1 and 2) with its
// additions in 96-bit integers.
//
// This GPU starts one FP64 addition of a warp every 19 cycles per SM but one
// 96-bit integer addition (three 32-bit ones with carries) every cycle, and the
// p = 2 transform is additions only.  A pass over a tile therefore turns its
// samples into fixed point once, runs all its stages exactly, and rounds once
// to FP64 on the way out.
//
// Precision.  The elements that a pass combines (a contiguous tile, or the rows
// of one column) share the exponent E of their largest.  Their 53-bit
// significands are placed 30 bits above the lowest, so that a pass's stages (12
// at most) cannot overflow 95 bits and a sign: elements down to 2^-30 of the
// largest enter exactly, smaller ones lose what lies below 2^-83 of it.
// Every result is the exact sum of those, rounded once, where FP64 stages round
// b times at 2^-53 of the partial sums.  The bits that were cut are fewer than
// 2^b units of the sum, so they matter only to a result below 2^(52+b) units (the
// large elements cancelled): a tile that has both is done again in levels, the
// cut remainders transformed in their own turn until nothing is left, and no
// result is off by more than 2^-52 of itself.  A tile with an infinity or a NaN
// runs the FP64 stages; results below the normal range go through one FP64 scaling.
//
// Tiles are 2^12 elements for 256 threads, 16 elements (48 words) each:
//   layout A  e = t + 256 r               bits 8..11 of the tile index in thread
//   layout C  e = 16 t + r                bits 0..3
//   layout B  e = (t & 15) + 16 r + 256 (t >> 4)    bits 4..7
// in that order, so that both ends move 128-byte runs.  The low pass takes the
// 12 low digits of a contiguous tile; a high pass of b digits has 2^b rows
// (2^d0 apart) of 2^(12-b) consecutive columns, its digits the top b bits of
// the tile index.
#include <algorithm>
#include <vector>

#include "dwt_internal.cuh"

namespace dwt {

namespace {

constexpr int kLT = 12;              // tile: 2^12 elements
constexpr int kNT = 256;             // threads, 16 elements each
constexpr int kPlane = (1 << kLT) + (1 << (kLT - 4));   // words of one limb's plane, one pad word per 16

struct DArgs {
    const double* in;
    double* out;
    long long ld_in, ld_out;
    long long S;        // row distance (high pass)
    int exp_shift;      // exponent of the factor: -m in the last pass of a forward transform
};

__device__ __forceinline__ int plane_pos(int e) { return e + (e >> 4); }

struct W96 {
    uint32_t a, b, c;   // low, middle, high word
};

__device__ __forceinline__ void bfly96(W96& x, W96& y) {
    W96 s, d;
    asm("add.cc.u32 %0, %3, %6;\n addc.cc.u32 %1, %4, %7;\n addc.u32 %2, %5, %8;"
        : "=r"(s.a), "=r"(s.b), "=r"(s.c)
        : "r"(x.a), "r"(x.b), "r"(x.c), "r"(y.a), "r"(y.b), "r"(y.c));
    asm("sub.cc.u32 %0, %3, %6;\n subc.cc.u32 %1, %4, %7;\n subc.u32 %2, %5, %8;"
        : "=r"(d.a), "=r"(d.b), "=r"(d.c)
        : "r"(x.a), "r"(x.b), "r"(x.c), "r"(y.a), "r"(y.b), "r"(y.c));
    x = s;
    y = d;
}

// negate when mask is all ones
__device__ __forceinline__ W96 negate_if(W96 v, uint32_t mask) {
    W96 r;
    asm("sub.cc.u32 %0, %3, %6;\n subc.cc.u32 %1, %4, %6;\n subc.u32 %2, %5, %6;"
        : "=r"(r.a), "=r"(r.b), "=r"(r.c)
        : "r"(v.a ^ mask), "r"(v.b ^ mask), "r"(v.c ^ mask), "r"(mask));
    return r;
}

__device__ __forceinline__ int exponent_of(uint32_t hi) { return (int)((hi >> 20) & 0x7ffu); }

constexpr int kG = 30;   // bits below the largest element's last place: 2^12 sums of 53 + 30 bits fit 95

// fixed point of a double against the largest exponent E (>= 1) of its group; cut:
// set if bits below the lowest are lost
__device__ __forceinline__ W96 to_fixed_any(uint32_t hi, uint32_t lo, int E, bool& cut) {
    const int ex = exponent_of(hi);
    uint32_t mh = hi & 0xfffffu;
    if (ex) mh |= 0x100000u;
    const int d = min(E - max(ex, 1), 95);
    if (d > kG) cut = cut || ((((unsigned long long)mh << 32) | lo) << (64 - min(d - kG, 64))) != 0;
    W96 v;   // significand << 30, then right by d
    v.a = lo << kG;
    v.b = __funnelshift_l(lo, mh, kG);
    v.c = mh >> (32 - kG);
    if (d >= 64) {
        v.a = v.c;
        v.b = v.c = 0;
    } else if (d >= 32) {
        v.a = v.b;
        v.b = v.c;
        v.c = 0;
    }
    const int r = d & 31;
    v.a = __funnelshift_r(v.a, v.b, r);
    v.b = __funnelshift_r(v.b, v.c, r);
    v.c >>= r;
    return negate_if(v, (uint32_t)((int)hi >> 31));
}

// the same for a normal double within 2^30 of E: one shift of the signed significand
__device__ __forceinline__ W96 to_fixed_near(uint32_t hi, uint32_t lo, int sh) {   // sh = 30 - E
    const uint32_t sign = (uint32_t)((int)hi >> 31);
    const int s = exponent_of(hi) + sh;
    uint32_t ml, mh;
    asm("sub.cc.u32 %0, %2, %4;\n subc.u32 %1, %3, %4;"
        : "=r"(ml), "=r"(mh)
        : "r"(lo ^ sign), "r"(((hi & 0xfffffu) | 0x100000u) ^ sign), "r"(sign));
    W96 v;
    v.a = ml << s;
    v.b = __funnelshift_l(ml, mh, s);
    v.c = __funnelshift_l(mh, sign, s);
    return v;
}

// the bits of a nonnegative v, normalised to bit 31 of h (lz places up), rounded
// to 53 (ties to even), with exponent field e of its top bit
__device__ __forceinline__ double round53(uint32_t h, uint32_t l, uint32_t rest, int e, uint32_t sign) {
    const uint32_t uh = h >> 11, ul = __funnelshift_r(l, h, 11);
    const uint32_t rem = (l & 0x7ffu) | (rest ? 1u : 0u);
    const uint32_t up = rem + (ul & 1u) > 0x400u ? 1u : 0u;
    uint32_t rl, rh;   // the implicit bit adds one to the exponent field
    asm("add.cc.u32 %0, %2, %3;\n addc.u32 %1, %4, %5;"
        : "=r"(rl), "=r"(rh)
        : "r"(ul), "r"(up), "r"(uh), "r"((uint32_t)(e - 1) << 20));
    return __hiloint2double((int)(rh | (sign & 0x80000000u)), (int)rl);
}

// fixed point of any size -> nearest double; top = exponent field of bit 95
__device__ __noinline__ double from_fixed_any(W96 v, uint32_t sign, int e) {   // v = |value|
    if (v.c == 0) {
        v.c = v.b;
        v.b = v.a;
        v.a = 0;
        e -= 32;
    }
    if (v.c == 0) {
        v.c = v.b;
        v.b = 0;
        e -= 32;
    }
    const int lz = __clz((int)v.c);   // 32 when the value is zero
    if (lz == 32) return 0.0;
    e -= lz;
    const uint32_t h = __funnelshift_l(v.b, v.c, lz), l = __funnelshift_l(v.a, v.b, lz), rest = v.a << lz;
    if (e >= 0x7ff) return __hiloint2double((int)(0x7ff00000u | (sign & 0x80000000u)), 0);
    if (e >= 1) return round53(h, l, rest, e, sign);
    return e + 128 < 1 ? 0.0 : round53(h, l, rest, e + 128, sign) * 0x1p-128;   // below the normal range
}

// fixed point -> nearest double (ties to even) of four numbers; top[i] = the
// exponent field of bit 95.  All lanes of the warp call it: results of normal
// size in the top word's range take the shortest way, and those in the second
// word's (below 2^-19 of the group's largest element, as high coefficients of
// smooth functions) the next one.
__device__ __forceinline__ void from_fixed4(const W96* v, const int* top, double* y) {
    uint32_t sign[4];
    W96 n[4];
    bool odd = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        sign[i] = (uint32_t)((int)v[i].c >> 31);
        n[i] = negate_if(v[i], sign[i]);
        odd = odd || n[i].c == 0 || (unsigned)(top[i] - 32) >= 0x7ffu - 32u;   // exponent 1 .. 0x7fe with up to 31 zeros
    }
    if (!__any_sync(0xffffffffu, odd)) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int lz = __clz((int)n[i].c);
            y[i] = round53(__funnelshift_l(n[i].b, n[i].c, lz), __funnelshift_l(n[i].a, n[i].b, lz), n[i].a << lz,
                           top[i] - lz, sign[i]);
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool z = n[i].c == 0;
        const uint32_t h = z ? n[i].b : n[i].c, l = z ? n[i].a : n[i].b, r = z ? 0u : n[i].a;
        const int lz = __clz((int)h), e = top[i] - lz - (z ? 32 : 0);
        if (__any_sync(0xffffffffu, h == 0 || (unsigned)(e - 1) >= 0x7feu))
            y[i] = from_fixed_any(n[i], sign[i], top[i]);
        else
            y[i] = round53(__funnelshift_l(l, h, lz), __funnelshift_l(r, l, lz), r << lz, e, sign[i]);
    }
}

// stages of register bits LO .. 3
template <int LO> __device__ __forceinline__ void stages(W96* v) {
#pragma unroll
    for (int i = 3; i >= LO; --i) {
#pragma unroll
        for (int r = 0; r < 16; ++r)
            if (!(r & (1 << i))) bfly96(v[r], v[r | (1 << i)]);
    }
}

__device__ __forceinline__ int e_a(int t, int r) { return t + kNT * r; }
__device__ __forceinline__ int e_c(int t, int r) { return 16 * t + r; }
__device__ __forceinline__ int e_b(int t, int r) { return (t & 15) + 16 * r + 256 * (t >> 4); }

template <int (*EL)(int, int)> __device__ __forceinline__ void put(uint32_t* p, const W96* v, int t) {
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int q = plane_pos(EL(t, r));
        p[q] = v[r].a;
        p[q + kPlane] = v[r].b;
        p[q + 2 * kPlane] = v[r].c;
    }
}
template <int (*EL)(int, int)> __device__ __forceinline__ void get(const uint32_t* p, W96* v, int t) {
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int q = plane_pos(EL(t, r));
        v[r].a = p[q];
        v[r].b = p[q + kPlane];
        v[r].c = p[q + 2 * kPlane];
    }
}

// |v| below 2^(52+B)
template <int B> __device__ __forceinline__ bool small96(const W96& v) {
    const W96 n = negate_if(v, (uint32_t)((int)v.c >> 31));
    if constexpr (B >= 12) return n.c == 0;
    else return n.c == 0 && n.b < (1u << (20 + B));
}

// element e of a tile in global memory
template <int B> __device__ __forceinline__ long long tile_off(int e, long long S) {
    constexpr int LC = kLT - B;
    return B == kLT ? (long long)e : (long long)(e & ((1 << LC) - 1)) + S * (long long)(e >> LC);
}

// A whole tile in levels: the part of every element that fits the fixed point of
// its group's largest is transformed exactly and taken off, then the next largest
// remainders, until none is left (each level's largest lies 2^-30 below the last
// one's at least).  Results add up in FP64 from the largest level down.
template <int B>
__device__ __noinline__ void tile_levels(const double* src, double* dst, long long S, int exp_shift, uint32_t* plane,
                                         int* emax) {
    constexpr int LC = kLT - B;
    const int t = threadIdx.x;
    const int top = 95 - 52 - kG + exp_shift;
    double x[16], y[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        x[r] = src[tile_off<B>(e_a(t, r), S)];
        y[r] = 0.0;
    }
    for (;;) {
        __syncthreads();   // the last level's exponents and planes have been read
        if (t < (1 << LC)) emax[t] = 1;
        __syncthreads();
        int mx = 1;
#pragma unroll
        for (int r = 0; r < 16; ++r) mx = max(mx, exponent_of((uint32_t)__double2hiint(x[r])));
        atomicMax(emax + (t & ((1 << LC) - 1)), mx);
        __syncthreads();
        const int E = emax[t & ((1 << LC) - 1)];
        W96 v[16];
        bool left = false;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const uint32_t hi = (uint32_t)__double2hiint(x[r]), lo = (uint32_t)__double2loint(x[r]);
            bool cut = false;
            v[r] = to_fixed_any(hi, lo, E, cut);
            if (cut) {   // the significand's low bits, exactly
                const int n = E - max(exponent_of(hi), 1) - kG;
                const unsigned long long keep = n >= 53 ? 0ull : ((((unsigned long long)hi << 32) | lo) >> n) << n;
                x[r] -= __longlong_as_double((long long)keep);
                left = true;
            } else {
                x[r] = 0.0;
            }
        }
        stages<0>(v);
        if constexpr (B > 4) {
            put<e_a>(plane, v, t);
            __syncthreads();
            if constexpr (B > 8) {
                get<e_c>(plane, v, t);
                stages<LC>(v);
                put<e_c>(plane, v, t);
                __syncthreads();
            }
            get<e_b>(plane, v, t);
            stages<(LC > 4 ? LC - 4 : 0)>(v);
        }
#pragma unroll
        for (int r = 0; r < 16; r += 4) {
            int tops[4];
            double z[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                tops[i] = emax[(B > 4 ? e_b(t, r + i) : e_a(t, r + i)) & ((1 << LC) - 1)] + top;
            from_fixed4(v + r, tops, z);
#pragma unroll
            for (int i = 0; i < 4; ++i) y[r + i] += z[i];
        }
        if (!__syncthreads_or(left)) break;
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) dst[tile_off<B>(B > 4 ? e_b(t, r) : e_a(t, r), S)] = y[r];
}

// One pass over 2^12-element tiles, B of the tile index's bits (the top ones)
// transformed: B = 12 the low pass, B < 12 a high pass with 2^(12-B) columns.
// Integer instructions bound it (ALU 72% busy at three CTAs per SM): per point 36
// of the additions, about 50 of the conversions and exchanges.  32 functions of
// 2^20 points: 1660 us on the FP64 pipe; so, with the
// short conversions 306 us, without groups of functions 270, with one vote per
// four results 256 (random values) and 274 (coefficients of a smooth function);
// with the votes on cut bits 255 .. 259 (m = 24, 2 functions 369 -> 374).
template <int B> __device__ __forceinline__ void pass_tile(const DArgs& a, long long tile, long long fn) {
    constexpr int LC = kLT - B;          // column bits
    extern __shared__ __align__(16) unsigned char smraw[];
    uint32_t* plane = reinterpret_cast<uint32_t*>(smraw);
    int* emax = reinterpret_cast<int*>(plane + 3 * kPlane);   // per column
    const int t = threadIdx.x;
    const long long nlo = a.S >> LC;     // tiles side by side below the pass's digits
    const long long base = B == kLT ? tile << kLT : ((tile % nlo) << LC) + (tile / nlo) * (a.S << B);
    const double* src = a.in + fn * a.ld_in + base;
    double* dst = a.out + fn * a.ld_out + base;
    auto off = [&](int e) { return tile_off<B>(e, a.S); };
    double x[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = src[off(e_a(t, r))];
    if constexpr (B <= 3) {
        // a few stages, all in thread: FP64
#pragma unroll
        for (int i = 3; i >= 4 - B; --i)
#pragma unroll
            for (int r = 0; r < 16; ++r)
                if (!(r & (1 << i))) {
                    const double p = x[r], q = x[r | (1 << i)];
                    x[r] = p + q;
                    x[r | (1 << i)] = p - q;
                }
        const double sc = __hiloint2double((1023 + a.exp_shift) << 20, 0);
#pragma unroll
        for (int r = 0; r < 16; ++r) dst[off(e_a(t, r))] = a.exp_shift ? x[r] * sc : x[r];
    } else {
        int mx = 1, mn = 0x7ff;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int ex = exponent_of((uint32_t)__double2hiint(x[r]));
            mx = max(mx, ex);
            mn = min(mn, ex);
        }
        if (t < (1 << LC)) emax[t] = 1;
        if (__syncthreads_or(mx == 0x7ff)) {
            // an infinity or a NaN: FP64 stages through shared memory
            double* y = reinterpret_cast<double*>(smraw);
#pragma unroll
            for (int r = 0; r < 16; ++r) y[e_a(t, r)] = x[r];
            for (int i = kLT - 1; i >= LC; --i) {
                __syncthreads();
                for (int q = t; q < (1 << (kLT - 1)); q += kNT) {
                    const int e0 = ((q >> i) << (i + 1)) | (q & ((1 << i) - 1)), e1 = e0 | (1 << i);
                    const double p = y[e0], s = y[e1];
                    y[e0] = p + s;
                    y[e1] = p - s;
                }
            }
            __syncthreads();
            const double sc = __hiloint2double((1023 + a.exp_shift) << 20, 0);
            for (int e = t; e < (1 << kLT); e += kNT) dst[off(e)] = y[e] * sc;
            return;
        }
        if constexpr (LC == 0) {
            mx = __reduce_max_sync(0xffffffffu, mx);
            if ((t & 31) == 0) atomicMax(emax, mx);
        } else {
            atomicMax(emax + (t & ((1 << LC) - 1)), mx);   // LC <= 8: a thread's elements share a column
        }
        __syncthreads();
        W96 v[16];
        bool cut = false;
        const int E = emax[t & ((1 << LC) - 1)];
        if (__all_sync(0xffffffffu, mn >= max(1, E - kG))) {
#pragma unroll
            for (int r = 0; r < 16; ++r)
                v[r] = to_fixed_near((uint32_t)__double2hiint(x[r]), (uint32_t)__double2loint(x[r]), kG - E);
        } else {
#pragma unroll
            for (int r = 0; r < 16; ++r)
                v[r] = to_fixed_any((uint32_t)__double2hiint(x[r]), (uint32_t)__double2loint(x[r]), E, cut);
        }
        const int top = 95 - 52 - kG + a.exp_shift;   // + E: exponent field of bit 95
        stages<0>(v);
        // nothing is written before this: bits cut and a result that would miss them
        auto missed = [&]() {
            bool lost = false;
#pragma unroll
            for (int r = 0; r < 16; ++r) lost = lost || small96<B>(v[r]);
            return __syncthreads_or(lost) != 0;
        };
        if constexpr (B == 4) {
            if (__syncthreads_or(cut) && missed()) return tile_levels<B>(src, dst, a.S, a.exp_shift, plane, emax);
#pragma unroll
            for (int r = 0; r < 16; r += 4) {
                const int tops[4] = {E + top, E + top, E + top, E + top};
                double y[4];
                from_fixed4(v + r, tops, y);
#pragma unroll
                for (int i = 0; i < 4; ++i) dst[off(e_a(t, r + i))] = y[i];
            }
        } else {
            put<e_a>(plane, v, t);
            const bool any_cut = __syncthreads_or(cut) != 0;
            if constexpr (B > 8) {
                get<e_c>(plane, v, t);
                stages<LC>(v);
                put<e_c>(plane, v, t);
                __syncthreads();
            }
            get<e_b>(plane, v, t);
            stages<(LC > 4 ? LC - 4 : 0)>(v);
            if (any_cut && missed()) return tile_levels<B>(src, dst, a.S, a.exp_shift, plane, emax);
#pragma unroll
            for (int r = 0; r < 16; r += 4) {
                int tops[4];
                double y[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) tops[i] = emax[e_b(t, r + i) & ((1 << LC) - 1)] + top;
                from_fixed4(v + r, tops, y);
#pragma unroll
                for (int i = 0; i < 4; ++i) dst[off(e_b(t, r + i))] = y[i];
            }
        }
    }
}

template <int B> __global__ void __launch_bounds__(kNT, 3) k2d_pass(DArgs a) {
    chain_begin();
    pass_tile<B>(a, blockIdx.x, blockIdx.y);
}

// One pass of several plans' transforms in one launch: job i owns the blocks
// [first, first + ntile * nf) (tile fastest), each of which runs the tile body of
// the plan's own launch.  LOW: the 12 low digits; else each job has its own digits.
// Lists of up to kGroupInline jobs travel in the launch's parameters.  32 jobs of
// 2^12 / 2^13 points: 127 / 242 us in launches of their own, 20 / 23 us so.
struct DGroup {
    DArgs a;
    int b;
    long long ntile, first;
};
constexpr int kGroupInline = 32;
struct DList {
    int n;
    const DGroup* far;   // n > kGroupInline
    DGroup near[kGroupInline];
};

template <bool LOW> __global__ void __launch_bounds__(kNT, 3) k2d_grouped(const __grid_constant__ DList list) {
    chain_begin();
    const DGroup* jobs = list.n > kGroupInline ? list.far : list.near;
    const long long blk = blockIdx.x;
    int lo = 0, hi = list.n - 1;   // the last job starting at or before this block
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].first <= blk) lo = mid;
        else hi = mid - 1;
    }
    const DArgs a = jobs[lo].a;
    const long long local = blk - jobs[lo].first, fn = local / jobs[lo].ntile, tile = local - fn * jobs[lo].ntile;
    if constexpr (LOW) {
        pass_tile<kLT>(a, tile, fn);
    } else {
        switch (jobs[lo].b) {
            case 1: pass_tile<1>(a, tile, fn); break;
            case 2: pass_tile<2>(a, tile, fn); break;
            case 3: pass_tile<3>(a, tile, fn); break;
            case 4: pass_tile<4>(a, tile, fn); break;
            case 5: pass_tile<5>(a, tile, fn); break;
            case 6: pass_tile<6>(a, tile, fn); break;
            case 7: pass_tile<7>(a, tile, fn); break;
            case 8: pass_tile<8>(a, tile, fn); break;
            default: pass_tile<9>(a, tile, fn); break;
        }
    }
}

constexpr size_t pass_smem(int b) { return b <= 3 ? 0 : (size_t)3 * kPlane * 4 + ((size_t)4 << (kLT - b)); }

template <int B> int launch_b(const DArgs& a, long long N, int nf, const char* fam, cudaStream_t st) {
    auto k = k2d_pass<B>;
    int rc = smem_limit_max(k);
    if (rc) return rc;
    {
        LaunchScope ls(fam, st);
        launch_chain(k, dim3((unsigned)(N >> kLT), (unsigned)nf), kNT, pass_smem(B), st, a);
    }
    DWT_CK_LAUNCH("k2d_pass");
    return DWT_OK;
}

int launch(int B, const DArgs& a, long long N, int nf, const char* fam, cudaStream_t st) {
    switch (B) {
        case 1: return launch_b<1>(a, N, nf, fam, st);
        case 2: return launch_b<2>(a, N, nf, fam, st);
        case 3: return launch_b<3>(a, N, nf, fam, st);
        case 4: return launch_b<4>(a, N, nf, fam, st);
        case 5: return launch_b<5>(a, N, nf, fam, st);
        case 6: return launch_b<6>(a, N, nf, fam, st);
        case 7: return launch_b<7>(a, N, nf, fam, st);
        case 8: return launch_b<8>(a, N, nf, fam, st);
        case 9: return launch_b<9>(a, N, nf, fam, st);
        case 12: return launch_b<12>(a, N, nf, fam, st);
        default: set_error("FP64 pass digits"); return DWT_EUNSUPPORTED;
    }
}

}  // namespace

bool p2d_ok(int m) { return m >= kLT; }

// high passes of a transform of 2^m points, and the digits of the k-th
static int high_passes(int m) { return (m - kLT + 8) / 9; }
static int high_digits(int m, int k) { return (m - kLT) / high_passes(m) + (k < (m - kLT) % high_passes(m) ? 1 : 0); }

// dwt_forward / dwt_inverse for p = 2, FP64, m >= 12: the 12 low digits, then
// the others in passes of at most 9 (rows of 64 bytes at least), as even as
// possible.  Each pass takes all functions: its conversions and additions bound
// it, not the traffic that groups of functions within L2 would save, and a
// group's last wave is short (32 functions of 2^20: 305 us in groups of 48 MB,
// 287 of 96 MB, 270 so; 8 of 2^22: 443, 416, 391; 2 of 2^24: 407, 407, 398).
int p2d_transform(dwt_plan_s* Pl, const double* in, double* out, int batch, long long ld_in, long long ld_out,
                  int sgn, cudaStream_t st) {
    const int m = Pl->m, nh = high_passes(m);
    const long long N = Pl->N;
    for (int f0 = 0; f0 < batch; f0 += 65535) {
        const int nf = std::min(65535, batch - f0);
        DArgs a{in + (long long)f0 * ld_in, out + (long long)f0 * ld_out, ld_in, ld_out, 1, 0};
        if (nh == 0 && sgn < 0) a.exp_shift = -m;
        int rc = launch(kLT, a, N, nf, "pass_lo", st);
        if (rc) return rc;
        int d = kLT;
        for (int k = 0; k < nh; ++k) {
            const int b = high_digits(m, k);
            DArgs h{out + (long long)f0 * ld_out, out + (long long)f0 * ld_out, ld_out, ld_out, 1ll << d, 0};
            if (k == nh - 1 && sgn < 0) h.exp_shift = -m;
            if ((rc = launch(b, h, N, nf, k == nh - 1 ? "pass_hi" : "pass_mid", st))) return rc;
            d += b;
        }
    }
    return DWT_OK;
}

// the transforms of several plans (p = 2, m >= 12, FP64): pass k of all jobs in one launch
int p2d_grouped(const std::vector<GroupJob>& jobs, int sgn, cudaStream_t st) {
    int most = 0;
    for (const GroupJob& j : jobs) most = std::max(most, 1 + high_passes(j.plan->m));
    std::vector<int> digit(jobs.size(), kLT);   // the next pass's first digit
    for (int k = 0; k < most; ++k) {
        std::vector<DGroup> h;
        long long blocks = 0;
        size_t smem = 0;
        for (size_t i = 0; i < jobs.size(); ++i) {
            const GroupJob& j = jobs[i];
            const int m = j.plan->m, nh = high_passes(m);
            if (k > nh) continue;
            DGroup g;
            g.b = k == 0 ? kLT : high_digits(m, k - 1);
            g.a = DArgs{(const double*)(k == 0 ? j.in : j.out), (double*)j.out, k == 0 ? j.ld_in : j.ld_out, j.ld_out,
                        k == 0 ? 1ll : 1ll << digit[i], k == nh && sgn < 0 ? -m : 0};
            if (k) digit[i] += g.b;
            g.ntile = j.plan->N >> kLT;
            g.first = blocks;
            blocks += g.ntile * j.batch;
            smem = std::max(smem, pass_smem(g.b));
            h.push_back(g);
        }
        if (blocks > 0x7fffffffll) {
            set_error("grouped FP64 pass: %lld blocks exceed one launch", blocks);
            return DWT_EINVAL;
        }
        auto kern = k == 0 ? k2d_grouped<true> : k2d_grouped<false>;
        int rc = smem_limit_max(kern);
        if (rc) return rc;
        DList list;
        list.n = (int)h.size();
        DGroup* d = nullptr;
        if (list.n > kGroupInline) {
            if (dmalloc((void**)&d, sizeof(DGroup) * h.size(), st)) return DWT_ENOMEM;
            DWT_CK(cudaMemcpyAsync(d, h.data(), sizeof(DGroup) * h.size(), cudaMemcpyHostToDevice, st));
        } else {
            std::copy(h.begin(), h.end(), list.near);
        }
        list.far = d;
        {
            LaunchScope ls("grouped_pass", st);
            launch_chain(kern, dim3((unsigned)blocks), kNT, smem, st, list);
        }
        dfree(d, st);
        DWT_CK_LAUNCH("k2d_grouped");
    }
    return DWT_OK;
}

}  // namespace dwt
