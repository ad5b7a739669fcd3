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

}  // namespace svk
