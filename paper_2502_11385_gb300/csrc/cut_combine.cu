// The contraction of a cut reconstruction on the fifth-generation tensor cores:
//   out[xb na + xa] = 2^-K sum_c U[c][xa] D[c][xb],  c < 4^K,
// as exact integer products of 8-bit digits.
//
// Every column of U (all codes of one xa) and of D is scaled by its own power of
// two to at most 1 and held as q = round(u 2^54), seven balanced digits:
// q = sum_i a_i 256^(6 - i), |a_0| <= 65, the others in [-128, 127], exact in
// float16.  The level sums z_L = sum_{i + j = L} sum_c a_i b_j, L <= 6, stay below
// 6.4e6 < 2^24 in magnitude for up to 64 codes (|z_L| <= 64 (L - 1) 2^14 +
// 64 * 2 * 65 * 128), and so does every partial sum: float32 accumulates them
// exactly in any order.  Left out are the levels beyond (below 2^-48 of the
// columns' largest product, some 2^-51 where the digits are random) and the
// rounding of q (2^-54 each); the float-pair contraction keeps 48 bits of each
// factor.
//
// A CTA takes tiles of 128 xa x 32 xb.  A (shared memory): the seven digit planes
// of 128 columns of U; B: those of 32 columns of D, one below the other, so that
// one MMA of digit i by B's first 7 - i planes adds to the accumulator columns of
// the levels i..6: N = 224, 192, ..., 32.  Two accumulators of 7 x 32 columns: the
// MMAs of a tile run while 16 warps read and join the one before (a seventeenth
// copies and issues: by one of the 16 the others waited for it at the barrier, 108 us), D's planes
// arrive by bulk copies two tiles ahead, U's stay for a row of tiles.
//
// What bounds it: joining seven words and forming a float64 without the FP64
// pipe (2 lanes a clock), some 60 instructions an output; the MMAs of a tile take
// 1792 clocks.  4096 x 4096 outputs of 64 codes: 82 us and 15 for the planes, where
// the float pairs on the FP32 units take 504; the error of the 40-qubit cut's
// distribution against 64 bits falls from 2.5e-14 of its norm to 4e-16.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "kernels.cuh"
#include "sv.h"
#include "tcgen05.cuh"

namespace svk {

namespace {

using namespace tc;

constexpr int kRows = 128, kCols = 32;   // tile: columns of U (TMEM lanes) and of D
constexpr int kLevels = 7;
constexpr int kJoin = 512;               // threads that read and join the accumulators
constexpr int kThreads = kJoin + 32;     // and a warp whose one lane copies and issues the MMAs
constexpr uint32_t kAccStep = 256;       // TMEM columns between the two accumulators

// K-elements (codes, padded to the MMA's 16) and bytes of a tile's digit planes.
__host__ __device__ constexpr int padded(int ncode) { return ncode < 16 ? 16 : ncode; }
__host__ __device__ constexpr uint32_t plane_a(int kp) { return (uint32_t)kp * kRows * 2; }
__host__ __device__ constexpr uint32_t bytes_a(int kp) { return kLevels * plane_a(kp); }
__host__ __device__ constexpr uint32_t bytes_b(int kp) { return (uint32_t)kp * kLevels * kCols * 2; }

// The columns x of U[code][x] and of D[code][x] to digit planes and exponents.  A CTA
// takes 32 columns (U's na first), eight codes a warp.  Core matrices of 8 rows x 8 codes (16 bytes a row): for U
// plane, 8 codes, row; for D 8 codes, then plane and row.
__global__ void __launch_bounds__(256) k_digit_planes(const double* __restrict__ U, const double* __restrict__ D,
                                                      int ncode, uint64_t na, uint64_t nb,
                                                      unsigned char* __restrict__ pa, unsigned char* __restrict__ pb,
                                                      int* __restrict__ ea, int* __restrict__ eb) {
    __shared__ int s_exp[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, kp = padded(ncode);
    const bool is_d = blockIdx.x >= na / 32;
    const uint64_t x = (uint64_t)blockIdx.x * 32 + lane - (is_d ? na : 0), nx = is_d ? nb : na;
    const double* __restrict__ src = is_d ? D : U;
    double v[8];
    int e = -2000;  // v < 2^e
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const int c = 8 * w + j;
        v[j] = c < ncode ? src[(uint64_t)c * nx + x] : 0.0;
        if (v[j] != 0.0) e = max(e, ilogb(v[j]) + 1);
    }
    s_exp[w][lane] = e;
    __syncthreads();
    for (int o = 0; o < 8; o++) e = max(e, s_exp[o][lane]);
    if (e == -2000) e = 0;
    if (w == 0) (is_d ? eb : ea)[x] = e;
    if (8 * w >= kp) return;
    unsigned short d[kLevels][8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
        long long q = __double2ll_rn(scalbn(v[j], 54 - e));
#pragma unroll
        for (int i = kLevels - 1; i > 0; i--) {
            const int a = (int)(((q & 255) ^ 128) - 128);
            q = (q - a) >> 8;
            d[i][j] = __half_as_ushort(__int2half_rn(a));
        }
        d[0][j] = __half_as_ushort(__int2half_rn((int)q));
    }
    const int rows = is_d ? kCols : kRows;
    unsigned char* tile = (is_d ? pb : pa) + (x / rows) * (uint64_t)(is_d ? bytes_b(kp) : bytes_a(kp));
    const int r = (int)(x % rows);
#pragma unroll
    for (int i = 0; i < kLevels; i++) {
        uint4 word;
        word.x = d[i][0] | (unsigned)d[i][1] << 16;
        word.y = d[i][2] | (unsigned)d[i][3] << 16;
        word.z = d[i][4] | (unsigned)d[i][5] << 16;
        word.w = d[i][6] | (unsigned)d[i][7] << 16;
        const uint32_t at = is_d ? (uint32_t)w * (kLevels * kCols * 16) + (uint32_t)(i * kCols + r) * 16
                                 : (uint32_t)i * plane_a(kp) + (uint32_t)w * (kRows * 16) + (uint32_t)r * 16;
        *reinterpret_cast<uint4*>(tile + at) = word;
    }
}

// t 2^x as a float64, rounded to nearest even, in integer arithmetic.
__device__ __forceinline__ double scaled(long long t, int x) {
    if (t == 0) return 0.0;
    const unsigned long long mag = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;
    const int lz = __clzll((long long)mag);
    const int e = 63 - lz + x + 1023;
    if (e <= 0) return scalbn((double)t, x);  // a subnormal result
    const unsigned long long n = mag << lz;
    unsigned long long m = n >> 11;  // 53 bits, the leading one among them
    const unsigned rem = (unsigned)n & 0x7ffu;
    m += (rem > 0x400u || (rem == 0x400u && (m & 1))) ? 1 : 0;
    const unsigned long long bits = ((unsigned long long)(e - 1) << 52) + m;
    return __longlong_as_double((long long)(bits | ((unsigned long long)t & 0x8000000000000000ull)));
}

__global__ void __launch_bounds__(kThreads, 1)
    k_combine_tc(const unsigned char* __restrict__ pa, const unsigned char* __restrict__ pb, const int* __restrict__ ea,
                 const int* __restrict__ eb, int kp, int n_cuts, uint64_t na, uint64_t nb, double* __restrict__ out,
                 int* __restrict__ fault) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t s_bar[5];  // full B 0, 1; full A; done 0, 1
    __shared__ uint32_t s_tmem;
    __shared__ int s_dead;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint64_t nbt = nb / kCols, tiles = (na / kRows) * nbt;
    const uint64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
    const uint32_t sa = smem_addr(sm), sb0 = sa + bytes_a(kp);
    auto full_b = [&](int b) { return smem_addr(&s_bar[b]); };
    const uint32_t full_a = smem_addr(&s_bar[2]);
    auto done = [&](int b) { return smem_addr(&s_bar[3 + b]); };
    auto sb = [&](int b) { return sb0 + b * bytes_b(kp); };
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(&s_tmem)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < 5; b++) mbar_init(smem_addr(&s_bar[b]), 1);
        s_dead = 0;
        fence_async_smem();
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem;
    int a_loads = 0, b_loads[2] = {0, 0};
    // one lane of the last warp copies and issues: A for the tile's U columns, B, the tile's MMAs
    auto load_a = [&](uint64_t t) {
        a_loads++;
        bulk_load(sa, pa + (t / nbt) * bytes_a(kp), bytes_a(kp), full_a);
    };
    auto load_b = [&](uint64_t t) {
        const int b = (int)(t - t0) & 1;
        b_loads[b]++;
        bulk_load(sb(b), pb + (t % nbt) * bytes_b(kp), bytes_b(kp), full_b(b));
    };
    auto issue = [&](uint64_t t) -> bool {
        const int b = (int)(t - t0) & 1;
        if (!wait(full_b(b), (uint32_t)((t - t0) >> 1) & 1, &s_dead)) return false;
        if (!wait(full_a, (uint32_t)(a_loads - 1) & 1, &s_dead)) return false;
        constexpr uint32_t step_a = kRows * 16, step_b = kLevels * kCols * 16;
        for (int k = 0; k < kp / 16; k++)
            for (int i = 0; i < kLevels; i++) {
                const uint64_t da = ((uint64_t)desc_hi(128) << 32) | desc_lo(sa + i * plane_a(kp) + 2 * k * step_a, step_a);
                const uint64_t db = ((uint64_t)desc_hi(128) << 32) | desc_lo(sb(b) + 2 * k * step_b, step_b);
                mma_smem(tmem + b * kAccStep + i * kCols, da, db, idesc(false, (kLevels - i) * kCols), k > 0 || i > 0);
            }
        commit(done(b));
        return true;
    };
    const bool boss = warp == kJoin / 32 && elect_one();
    bool ok = true;  // that lane: its waits came to their end
    if (boss && t0 < t1) {
        load_a(t0);
        load_b(t0);
        if (t0 + 1 < t1) load_b(t0 + 1);
        ok = issue(t0);
        if (!ok) s_dead = 1;
    }
    uint64_t issued = ok ? t0 + 1 : t0;  // tiles whose MMAs it has issued
    const int r0 = (warp >> 2) * 8;
    int failed = 0;
    for (uint64_t t = t0; t < t1; t++) {
        const int b = (int)(t - t0) & 1;
        const bool same_a = t + 1 < t1 && (t + 1) / nbt == t / nbt;
        if (boss && ok && same_a) {
            ok = issue(t + 1);
            issued += ok ? 1 : 0;
        }
        bool bad = !wait(done(b), (uint32_t)((t - t0) >> 1) & 1, &s_dead);
        fence_after();
        if (boss && ok) {
            if (t + 2 < t1) load_b(t + 2);  // the tile's MMAs have read B
            if (t + 1 < t1 && !same_a) {    // and A
                load_a(t + 1);
                ok = issue(t + 1);
                issued += ok ? 1 : 0;
            }
        }
        bad = bad || !ok;
        if (bad) s_dead = 1;
        __syncwarp();
        if (warp < kJoin / 32) {
            const uint64_t xa = (t / nbt) * kRows + (warp & 3) * 32 + lane, xb0 = (t % nbt) * kCols + r0;
            uint32_t z[kLevels][8];
#pragma unroll
            for (int l = 0; l < kLevels; l++)
                ldN<8>(tmem + b * kAccStep + l * kCols + r0 + ((uint32_t)(warp & 3) << 21), z[l]);
            ld_wait();
            fence_before();
            const int xa_exp = ea[xa] - 52 - n_cuts;
#pragma unroll
            for (int j = 0; j < 8; j++) {
                int v[kLevels];
#pragma unroll
                for (int l = 0; l < kLevels; l++) v[l] = __float2int_rn(__uint_as_float(z[l][j]));
                const long long sum = ((long long)(v[0] * 256 + v[1]) << 32) + ((long long)(v[2] * 256 + v[3]) << 16) +
                                      (v[4] * 256 + v[5]) + ((v[6] + 128) >> 8);
                out[(xb0 + j) * na + xa] = scaled(sum, xa_exp + eb[xb0 + j]);
            }
        }
        failed = __syncthreads_or(bad);  // the accumulator is free
        fence_after();
        if (failed) break;
    }
    if (boss && failed) {
        // the copies and MMAs still in flight, once more within the limits
        *fault = 1;
        volatile int none = 0;
        (void)wait(full_a, (uint32_t)(a_loads - 1) & 1, &none);
        for (int b = 0; b < 2; b++) {
            if (b_loads[b]) (void)wait(full_b(b), (uint32_t)(b_loads[b] - 1) & 1, &none);
            if (issued > t0 + b) (void)wait(done(b), (uint32_t)((issued - 1 - t0 - b) >> 1) & 1, &none);
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512) : "memory");
    }
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

// Up to 64 codes (the level sums' bound), whole tiles, and 2^20 outputs: there the planes and this
// kernel take 24 us (64 codes; 18 of them with 4), the float pairs 36 and 21 for half as many, and
// below the launches count.
size_t combine_tc_bytes(int n_cuts, uint64_t na, uint64_t nb) {
    if (n_cuts > 3 || na < kRows || nb < kCols || na * nb < (1ull << 20)) return 0;
    const int kp = padded(1 << (2 * n_cuts));
    return 256 + align256(4 * na) + align256(4 * nb) + align256(na / kRows * bytes_a(kp)) +
           align256(nb / kCols * bytes_b(kp));
}

cudaError_t launch_combine_tc(const double* U, const double* D, int n_cuts, uint64_t na, uint64_t nb, double* out,
                              void* scratch, int sms, cudaStream_t s) {
    const int ncode = 1 << (2 * n_cuts), kp = padded(ncode);
    auto* fault = (int*)scratch;
    unsigned char* p = (unsigned char*)scratch + 256;
    auto* ea = (int*)p;
    p += align256(4 * na);
    auto* eb = (int*)p;
    p += align256(4 * nb);
    unsigned char* pa = p;
    unsigned char* pb = p + align256(na / kRows * bytes_a(kp));
    const uint32_t smem = std::max(bytes_a(kp) + 2 * bytes_b(kp), 116u * 1024);  // one CTA per SM (its tensor memory)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    static std::atomic<bool> ready[64];
    if (e == cudaSuccess && !ready[dev].load()) {
        e = cudaFuncSetAttribute(k_combine_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(bytes_a(64) + 2 * bytes_b(64)));
        if (e == cudaSuccess) ready[dev].store(true);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(fault, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    k_digit_planes<<<(unsigned)(na / 32 + nb / 32), 256, 0, s>>>(U, D, ncode, na, nb, pa, pb, ea, eb);
    const uint64_t tiles = (na / kRows) * (nb / kCols);
    k_combine_tc<<<(unsigned)std::min<uint64_t>(tiles, (uint64_t)sms), kThreads, smem, s>>>(pa, pb, ea, eb, kp, n_cuts,
                                                                                          na, nb, out, fault);
    return cudaGetLastError();
}

}  // namespace svk
