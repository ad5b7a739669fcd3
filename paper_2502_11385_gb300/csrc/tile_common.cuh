// Device helpers shared by the tile-pass kernels.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "device_types.hpp"

namespace svk {

template <typename R>
struct alignas(2 * sizeof(R)) Cx {
    R re, im;
};

__device__ __forceinline__ float fmaT(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return fma(a, b, c); }

// ---------------------------------------------------------------------------
// Shared-memory layout of a tile: 16-byte slots, XOR-swizzled so that warps
// gathering amplitudes at power-of-two strides spread over the banks.
// ---------------------------------------------------------------------------
// swz(j) = j ^ L(j) with L linear over GF(2) (shifts and XORs), so
// swz(a ^ b) = swz(a) ^ swz(b).
template <typename R>
__device__ __forceinline__ int swz(int j) {
    constexpr int VS = (sizeof(R) == 4) ? 1 : 0;  // log2(amplitudes per 16-byte slot); R = float or double
    int s = j >> VS;
    int h = (s >> 3) ^ (s >> 6) ^ (s >> 9) ^ (s >> 12);
    s ^= h & 7;
    return (s << VS) | (j & ((1 << VS) - 1));
}

// Diagonal ops visit amplitude i = t + it * 2^LT for thread t of 2^LT.  The
// phase-table index takes bit j from tile position pos[j] (or, for a
// non-local qubit, from the tile's base index); the bits below log2 of the
// CTA size come from the thread id and are gathered once per op.
struct DiagIndex {
    int idx_t;  // table-index bits fixed for this thread
    int hp;     // 5 bits per table bit j: its tile position relative to the CTA size, or 31
    int sw_t;   // swizzle of the thread's part of i
};

template <typename SwzT, int LT = 8>  // LT = log2 of the CTA size
__device__ __forceinline__ DiagIndex diag_index(const DevOp& op, uint64_t tile_base, int t) {
    DiagIndex d;
    d.idx_t = 0;
    d.hp = 0;
#pragma unroll
    for (int j = 0; j < 5; j++) {
        int h = 31;  // (it >> 31) & 1 = 0: the bit is not taken from it
        if (j < op.k) {
            const int p = op.pos[j];
            if (p < 0) d.idx_t |= (int)((tile_base >> op.qbit[j]) & 1) << j;
            else if (p < LT) d.idx_t |= ((t >> p) & 1) << j;
            else h = p - LT;
        }
        d.hp |= h << (5 * j);
    }
    d.sw_t = swz<SwzT>(t);
    return d;
}

template <typename SwzT, int LT = 8>
__device__ __forceinline__ void diag_at(const DiagIndex& d, int it, int& idx, int& sidx) {
    idx = d.idx_t;
#pragma unroll
    for (int j = 0; j < 5; j++) idx |= ((it >> ((d.hp >> (5 * j)) & 31)) & 1) << j;
    sidx = d.sw_t ^ swz<SwzT>(it << LT);
}

// Applies a <- f(u, a) to every amplitude of the tile (u its phase-table
// entry), U amplitudes of a thread at a time: their loads are all issued
// before their stores, so the U table and tile reads overlap.
template <int U, int LT, typename SwzT, typename T, typename E, typename F>
__device__ __forceinline__ void diag_sweep(T* sm, int m, const DiagIndex& d, int t, const E* M, F f) {
    const int N = 1 << m;
    if (N >= (1 << LT)) {
        const int iters = N >> LT;
        int it = 0;
        for (; it + U <= iters; it += U) {
            int idx[U], si[U];
            E u[U];
            T a[U];
#pragma unroll
            for (int q = 0; q < U; q++) diag_at<SwzT, LT>(d, it + q, idx[q], si[q]);
#pragma unroll
            for (int q = 0; q < U; q++) {
                u[q] = M[idx[q]];
                a[q] = sm[si[q]];
            }
#pragma unroll
            for (int q = 0; q < U; q++) sm[si[q]] = f(u[q], a[q]);
        }
        for (; it < iters; it++) {
            int idx, si;
            diag_at<SwzT, LT>(d, it, idx, si);
            sm[si] = f(M[idx], sm[si]);
        }
    } else if (t < N) {  // a tile smaller than the CTA: threads past N idle
        int idx, si;
        diag_at<SwzT, LT>(d, 0, idx, si);
        sm[si] = f(M[idx], sm[si]);
    }
}

template <typename T>
__device__ __forceinline__ T rot_i(T v, int code) {  // v * i^code for {re, im} pairs
    using E = decltype(v.re);
    const E re = v.re, im = v.im;
    if (code == 1) return T{-im, re};
    if (code == 2) return T{-re, -im};
    if (code == 3) return T{im, -re};
    return v;
}

struct alignas(16) Q2 {
    long long re, im;
};
__device__ __forceinline__ Q2 rot_q(Q2 v, int c) { return rot_i(v, c); }  // exact: |re|, |im| < 2^63

// float64 -> fixed point with FB fraction bits (x * 2^FB truncated toward
// zero), for |x| < 2^(62 - FB) (components of a normalised state): the
// significand with its implicit bit is placed at bits 62..10 and shifted
// right by 1023 - exponent + 62 - FB; zero and subnormal inputs (shift
// clamped at 63) give 0.  Branch-free.
template <int FB = 62>
__device__ __forceinline__ long long d2q(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const int s = min(max(1023 + 62 - FB - (int)((hi >> 20) & 0x7FFu), 0), 63);
    const unsigned mh = (__funnelshift_l(lo, hi, 10) & 0x3FFFFFFFu) | 0x40000000u;
    const long long v = (long long)((((unsigned long long)mh << 32) | (unsigned long long)(lo << 10)) >> s);
    return (int)hi < 0 ? -v : v;
}

// Fixed point with FB fraction bits -> float64, truncated toward zero: |q|
// normalised by its leading-zero count, the 52 bits below the leading one
// form the fraction.
template <int FB = 62>
__device__ __forceinline__ double q2d(long long q) {
    const unsigned long long sign = (unsigned long long)q & 0x8000000000000000ull;
    const unsigned long long a = sign ? 0ull - (unsigned long long)q : (unsigned long long)q;
    const int lz = __clzll((long long)a);
    const unsigned long long n = a << (lz & 63);                      // leading one at bit 63 (a != 0)
    const unsigned long long E = (unsigned long long)(1086 - FB - lz);  // value = a * 2^-FB
    const unsigned long long bits = sign | (E << 52) | ((n >> 11) & ((1ull << 52) - 1));
    return __longlong_as_double(a ? (long long)bits : 0ll);
}

// (a * b) >> 62, floor: Q62 x Q62 -> Q62, or a Q62 phase times a Q56
// amplitude -> Q56
__device__ __forceinline__ long long qmul(long long a, long long b) {
    const long long hi = __mul64hi(a, b);
    const unsigned long long lo = (unsigned long long)(a * b);
    return (long long)(((unsigned long long)hi << 2) | (lo >> 62));
}

// ---------------------------------------------------------------------------
// K5-df: tile pass for complex128 states with double-float arithmetic.
//
// GB300's FP64 units run about 70x slower than its FP32 units, so complex128
// gates are computed on (hi, lo) float pairs instead (Dekker 1971): each
// float64 amplitude component is split once per pass, when the tile is
// loaded, into hi = its leading 24 significant bits and lo = the next 23
// (47 bits, |x - hi - lo| <= 2^-47 |x|), with integer bit operations so the
// FP64 pipe stays idle; block products use error-free TwoProd (FMA) and
// TwoSum transforms (the compensated dot product of Ogita, Rump and Oishi
// 2005, with double-float inputs); the tile is re-assembled into float64 on
// store, again with integer operations.
// ---------------------------------------------------------------------------
struct alignas(16) DF4 {
    float rh, rl, ih, il;  // re = rh + rl, im = ih + il
};
__device__ __forceinline__ DF4 rot_df(DF4 v, int c) {  // v * i^c
    if (c == 1) return DF4{-v.ih, -v.il, v.rh, v.rl};
    if (c == 2) return DF4{-v.rh, -v.rl, -v.ih, -v.il};
    if (c == 3) return DF4{v.ih, v.il, -v.rh, -v.rl};
    return v;
}

__device__ __forceinline__ void d2df(double x, float& h, float& l) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi32 = (unsigned)(b >> 32), lo32 = (unsigned)b;
    const unsigned sign = hi32 & 0x80000000u;
    const int e = (int)((hi32 >> 20) & 0x7ff);
    if (e < 897) {  // |x| < 2^-126 (or zero): below float's normal range, dropped
                    // (for 2^-126 <= |x| < 2^-103 only hi is kept: absolute error < 2^-126)
        h = 0.f;
        l = 0.f;
        return;
    }
    // amplitudes satisfy |x| <= 1 < 2^127, so e - 896 fits float's exponent field
    h = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | ((hi32 & 0xFFFFFu) << 3) | (lo32 >> 29));
    const unsigned r = (lo32 >> 6) & 0x7FFFFFu;  // next 23 mantissa bits, weight 2^(e-1069)
    const int B = e - 919;                       // float exponent field with 2^(B-150) = 2^(e-1069)
    if (B < 1 || r == 0u) {
        l = 0.f;
        return;
    }
    const unsigned one = sign | ((unsigned)B << 23);
    l = __fadd_rn(__uint_as_float(one | r), -__uint_as_float(one));  // exact: (1 + r 2^-23) 2^(B-127) - 2^(B-127)
}

__device__ __forceinline__ double df2d(float h, float l) {
    const float s = __fadd_rn(h, l);  // Fast2Sum: |l| <= ulp(s)/2 afterwards
    l = __fadd_rn(l, -__fadd_rn(s, -h));
    h = s;
    const unsigned hb = __float_as_uint(h);
    const unsigned eh = (hb >> 23) & 0xffu;
    if (eh == 0u) return 0.0;  // zero or subnormal hi: below the amplitudes' range
    const unsigned long long D = ((unsigned long long)(hb & 0x80000000u) << 32) |
                                 ((unsigned long long)(eh + 896u) << 52) |
                                 ((unsigned long long)(hb & 0x7FFFFFu) << 29);
    const unsigned lb = __float_as_uint(l);
    if ((lb & 0x7FFFFFFFu) == 0u) return __longlong_as_double((long long)D);
    // l = ml * 2^(el - 150) (subnormal l: no implicit bit, el taken as 1)
    const unsigned el_raw = (lb >> 23) & 0xffu;
    const unsigned el = el_raw ? el_raw : 1u;
    const unsigned long long ml = (unsigned long long)((lb & 0x7FFFFFu) | (el_raw ? 0x800000u : 0u));
    // in units of ulp_double(h) = 2^(eh - 179): k = ml * 2^(el - eh + 29), el <= eh - 24
    const int sh = (int)el - (int)eh + 29;
    unsigned long long k = sh >= 0 ? (ml << sh) : (sh > -40 ? (ml >> (-sh)) : 0ull);
    unsigned long long mag = D & 0x7FFFFFFFFFFFFFFFull;
    if ((lb ^ hb) & 0x80000000u) {
        if ((hb & 0x7FFFFFu) == 0u) k <<= 1;  // hi is a power of two: the result lies in the lower binade
        mag -= k;
    } else {
        mag += k;  // no carry out of the mantissa: |l| <= 2^28 ulp_double(h)
    }
    return __longlong_as_double((long long)((D & 0x8000000000000000ull) | mag));
}

// (sh, sl) += x * y for double-floats x = (xh, xl), y = (yh, yl): TwoProd of the
// high parts, first-order cross terms, TwoSum into the running sum.  __fmul_rn
// and __fadd_rn keep the compiler from contracting the transforms into FMAs.
__device__ __forceinline__ void df_mac(float& sh, float& sl, float xh, float xl, float yh, float yl) {
    const float ph = __fmul_rn(xh, yh);
    const float pe = fmaf(xh, yh, -ph);
    const float pl = fmaf(xh, yl, fmaf(xl, yh, pe));
    const float s = __fadd_rn(sh, ph);
    const float bb = __fadd_rn(s, -sh);
    const float err = __fadd_rn(__fadd_rn(sh, -__fadd_rn(s, -bb)), __fadd_rn(ph, -bb));
    sh = s;
    sl = __fadd_rn(sl, __fadd_rn(err, pl));
}

__device__ __forceinline__ void df_norm(float& h, float& l) {
    const float s = __fadd_rn(h, l);
    l = __fadd_rn(l, -__fadd_rn(s, -h));
    h = s;
}

// (sh, sl) = x * y as an unnormalised double-float (TwoProd + cross terms).
__device__ __forceinline__ void df_mul(float& sh, float& sl, float xh, float xl, float yh, float yl) {
    sh = __fmul_rn(xh, yh);
    sl = fmaf(xh, yl, fmaf(xl, yh, fmaf(xh, yh, -sh)));
}

}  // namespace svk
