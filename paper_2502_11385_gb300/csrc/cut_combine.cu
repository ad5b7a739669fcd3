// The contraction of a cut reconstruction on the fifth-generation tensor cores:
//   out[xb na + xa] = 2^-K sum_c U[c][xa] D[c][xb],  c < 4^K,
// as exact integer products of 8-bit digits.
//
// Every column of U (all codes of one xa) and of D is scaled by its own power of
// two, 2^ea or 2^eb, to below 1 and held as q = round(u 2^62), eight balanced
// digits: q = sum_i a_i 256^(7 - i), |a_0| <= 65, the others in [-128, 127], exact
// in float16.  The level sums z_L = sum_{i + j = L} sum_c a_i b_j, L <= 7, stay
// below 7.4e6 < 2^24 in magnitude for up to 64 codes (|z_L| <= 64 (L - 1) 2^14 +
// 64 * 2 * 65 * 128), and so does every partial sum: float32 accumulates them
// exactly in any order.
//
// Error, in units of 2^(ea + eb - K): at most 4^K 7.03 2^-62 from the levels left
// out, 4^K 2^-62 from rounding q (entries below 2^-9 of their column's largest only),
// 2^-57 where the levels are joined; 4^K 2^-58.9 + 2^-57 in all, then the result's own
// rounding.  The float pairs' error is in proportion to sum_c |U_c D_c| (random codes:
// 2^-48.5 of it rms for one cut, 2^-47.6 for two, 2^-46.1 for three, and some 2^-45.2,
// 2^-44.3, 2^-42.4 at most), and the two scales say nothing of that sum where a column's
// large codes meet small ones of the other (outcomes that are correlated across the cut:
// beside an outcome of weight 1 the probabilities of one of 2^-30 kept 20 bits).  So a
// column is marked with the codes that lie within 2^kGap of its scale.  One marked in both
// columns makes the sum at least 2^-10 of the scales' product and the error at most
// 2^-46.0, 2^-44.6 or 2^-42.8 of it (2^-48.5 rms); no code that is not 0 in both makes the
// output exactly 0.  Any other output is formed anew from float pairs of the scaled codes,
// by the warp that holds it: the same sums, in the same order, as k_combine (cut.cu).  A
// warp first looks at the marks that all its 32 x 8 outputs share.
//
// A CTA takes tiles of 128 xa x 32 xb.  A (shared memory): the eight digit planes
// of 128 columns of U; B: those of 32 columns of D, one below the other, so that
// one MMA of digit i by B's first 8 - i planes adds to the accumulator columns of
// the levels i..7: N = 256, 224, ..., 32.  Two accumulators of 8 x 32 columns: the
// MMAs of a tile run while 16 warps read and join the one before (a seventeenth
// copies and issues: by one of the 16 the others waited for it at the barrier, 108 us), D's planes
// arrive by bulk copies two tiles ahead, U's stay for a row of tiles.
//
// What bounds it: joining eight words and forming a float64 without the FP64
// pipe (2 lanes a clock), some 60 instructions an output; the MMAs of a tile take
// 2304 clocks.  4096 x 4096 outputs of 64 codes: 97 us and 11 for the planes (seven
// digits without the marks took 82 and 15), where the float pairs on the FP32 units
// take 504; the error of the 40-qubit cut's distribution against 64 bits falls from
// 2.5e-14 of its norm to 4e-16 or less.  Where every output goes to the pairs (no
// column's large codes meet large ones) the pairs take some 650: calls of one, two and
// three cuts 455, 655 and 1509 us, with k_combine 814, 1002 and 1350.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "float_pair.cuh"
#include "kernels.cuh"
#include "sv.h"
#include "tcgen05.cuh"
#include "tile_common.cuh"

namespace svk {

namespace {

using namespace tc;

constexpr int kRows = 128, kCols = 32;   // tile: columns of U (TMEM lanes) and of D
constexpr int kLevels = 8;
constexpr int kUnit = 56;                // the joined levels count units of 2^-56
constexpr int kGap = 5;                  // log2 below its column's scale of a code that is marked as large
constexpr int kJoinCols = 8;             // columns of D that a joining thread takes
constexpr int kJoin = 512;               // threads that read and join the accumulators
constexpr int kThreads = kJoin + 32;     // and a warp whose one lane copies and issues the MMAs
constexpr uint32_t kAccStep = 256;       // TMEM columns between the two accumulators

// K-elements (codes, padded to the MMA's 16) and bytes of a tile's digit planes.
__host__ __device__ constexpr int padded(int ncode) { return ncode < 16 ? 16 : ncode; }
__host__ __device__ constexpr uint32_t plane_a(int kp) { return (uint32_t)kp * kRows * 2; }
__host__ __device__ constexpr uint32_t bytes_a(int kp) { return kLevels * plane_a(kp); }
__host__ __device__ constexpr uint32_t bytes_b(int kp) { return (uint32_t)kp * kLevels * kCols * 2; }

// A column's codes within 2^kGap of its scale, and those that are not 0.
struct alignas(16) Marks {
    unsigned long long large, some;
};

// The columns x of U[code][x] and of D[code][x] to digit planes, exponents and marks; the
// scaled values themselves become float pairs, in place.  A CTA takes 32 columns (U's na first),
// eight codes a warp.  Core matrices of 8 rows x 8 codes (16 bytes a row): for U
// plane, 8 codes, row; for D 8 codes, then plane and row.
__global__ void __launch_bounds__(256) k_digit_planes(double* __restrict__ U, double* __restrict__ D,
                                                      int ncode, uint64_t na, uint64_t nb,
                                                      unsigned char* __restrict__ pa, unsigned char* __restrict__ pb,
                                                      int* __restrict__ ea, int* __restrict__ eb,
                                                      Marks* __restrict__ ma, Marks* __restrict__ mb) {
    __shared__ int s_exp[8][32];
    __shared__ unsigned char s_large[32][8], s_some[32][8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, kp = padded(ncode);
    const bool is_d = blockIdx.x >= na / 32;
    const uint64_t x = (uint64_t)blockIdx.x * 32 + lane - (is_d ? na : 0), nx = is_d ? nb : na;
    double* __restrict__ src = is_d ? D : U;
    constexpr int kNone = -2000;
    double v[8];
    int ex[8], e = kNone;  // 2^(ex - 1) <= |v| < 2^ex (terms are multiples of 2^-112: none is subnormal), |v| < 2^e
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const int c = 8 * w + j;
        v[j] = c < ncode ? src[(uint64_t)c * nx + x] : 0.0;
        ex[j] = v[j] != 0.0 ? (__double2hiint(v[j]) >> 20 & 0x7ff) - 1022 : kNone;
        e = max(e, ex[j]);
    }
    s_exp[w][lane] = e;
    __syncthreads();
    for (int o = 0; o < 8; o++) e = max(e, s_exp[o][lane]);
    unsigned large = 0, some = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        some |= (ex[j] != kNone ? 1u : 0u) << j;
        large |= (ex[j] != kNone && ex[j] > e - kGap ? 1u : 0u) << j;  // |v| >= 2^(e - kGap)
    }
    s_large[lane][w] = (unsigned char)large;
    s_some[lane][w] = (unsigned char)some;
    __syncthreads();
    if (e == kNone) e = 0;
    if (w == 0) {
        (is_d ? eb : ea)[x] = e;
        Marks m{0, 0};
        for (int o = 7; o >= 0; o--) {
            m.large = m.large << 8 | s_large[lane][o];
            m.some = m.some << 8 | s_some[lane][o];
        }
        (is_d ? mb : ma)[x] = m;
    }
    if (8 * w >= kp) return;
    unsigned short d[kLevels][8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const int c = 8 * w + j;
        const double u = ex[j] == kNone ? 0.0 : __hiloint2double(__double2hiint(v[j]) - (e << 20), __double2loint(v[j]));
        if (c < ncode) reinterpret_cast<float2*>(src)[(uint64_t)c * nx + x] = pair_of(u);
        // 53 bits, shifted left by 9 - (e - ex), or right and rounded
        const unsigned long long bits = (unsigned long long)__double_as_longlong(u);
        const unsigned long long mant = (bits & ((1ull << 52) - 1)) | 1ull << 52;
        const int down = e - ex[j] - 9;
        long long q = ex[j] == kNone || down > 53 ? 0
                      : down <= 0                 ? (long long)(mant << -down)
                                                  : (long long)((mant + (1ull << (down - 1))) >> down);
        q = v[j] < 0.0 ? -q : q;
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

__device__ __forceinline__ unsigned long long shared_marks(unsigned long long m) {  // by all lanes of the warp
    return (unsigned long long)__reduce_and_sync(~0u, (unsigned)(m >> 32)) << 32 | __reduce_and_sync(~0u, (unsigned)m);
}

// (s + c) 2^x as a float64, truncated, in integer arithmetic (the result is normal or 0).
__device__ __forceinline__ double pair_scaled(float s, float c, int x) {
    const float h = __fadd_rn(s, c), z = __fsub_rn(h, s);
    const float l = __fadd_rn(__fsub_rn(s, __fsub_rn(h, z)), __fsub_rn(c, z));  // s + c = h + l exactly
    const double d = df2d(h, l);
    return d == 0.0 ? 0.0 : __hiloint2double(__double2hiint(d) + (x << 20), __double2loint(d));
}

// The outputs of column xa by columns xb0.. of D whose bits are set in `which`, from float
// pairs.
__device__ __forceinline__ void by_pairs(const float2* __restrict__ U, const float2* __restrict__ D, int ncode,
                                         uint64_t na, uint64_t nb, uint64_t xa, uint64_t xb0, unsigned which, int xa_exp,
                                         const int* __restrict__ eb, double* __restrict__ out) {
    constexpr int kBatch = 2, kVec = kJoinCols / 2;  // codes (of 4^K) whose loads are in flight together
    float s[kJoinCols], c[kJoinCols];
#pragma unroll
    for (int j = 0; j < kJoinCols; j++) s[j] = c[j] = 0.f;
    const float2* u = U + xa;
    const float4* d = reinterpret_cast<const float4*>(D + xb0);
#pragma unroll 1
    for (int left = ncode; left > 0; left -= kBatch) {
        float2 x[kBatch];
        float4 y[kBatch][kVec];
#pragma unroll
        for (int i = 0; i < kBatch; i++, u += na, d += nb / 2) {
            x[i] = *u;
#pragma unroll
            for (int j = 0; j < kVec; j++) y[i][j] = d[j];
        }
#pragma unroll
        for (int i = 0; i < kBatch; i++)
#pragma unroll
            for (int j = 0; j < kVec; j++) {
                dot2_add(s[2 * j], c[2 * j], x[i], make_float2(y[i][j].x, y[i][j].y));
                dot2_add(s[2 * j + 1], c[2 * j + 1], x[i], make_float2(y[i][j].z, y[i][j].w));
            }
    }
#pragma unroll
    for (int j = 0; j < kJoinCols; j++)
        if (which >> j & 1) out[(xb0 + j) * na + xa] = pair_scaled(s[j], c[j], xa_exp + eb[xb0 + j]);
}

__global__ void __launch_bounds__(kThreads, 1)
    k_combine_tc(const unsigned char* __restrict__ pa, const unsigned char* __restrict__ pb, const int* __restrict__ ea,
                 const int* __restrict__ eb, const Marks* __restrict__ ma, const Marks* __restrict__ mb,
                 const float2* __restrict__ U, const float2* __restrict__ D, int n_cuts, uint64_t na, uint64_t nb,
                 double* __restrict__ out, int* __restrict__ fault) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t s_bar[5];  // full B 0, 1; full A; done 0, 1
    __shared__ uint32_t s_tmem;
    __shared__ int s_dead;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ncode = 1 << (2 * n_cuts), kp = padded(ncode);
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
    const int r0 = (warp >> 2) * kJoinCols;
    int failed = 0;
    uint64_t row = ~0ull;               // the row of tiles of
    unsigned long long large = 0, all_a = 0;  // large codes: this thread's column of U, all the warp's
    // of the column of D of lane % 8, the next tile's
    auto large_b = [&](uint64_t t) { return mb[(t % nbt) * kCols + r0 + (lane & (kJoinCols - 1))].large; };
    unsigned long long ahead = warp < kJoin / 32 && t0 < t1 ? large_b(t0) : 0;
    for (uint64_t t = t0; t < t1; t++) {
        const int b = (int)(t - t0) & 1;
        const bool same_a = t + 1 < t1 && (t + 1) / nbt == t / nbt;
        if (boss && ok && same_a) {
            ok = issue(t + 1);
            issued += ok ? 1 : 0;
        }
        unsigned rest = 0;  // the thread's outputs that the scales do not bound
        if (warp < kJoin / 32) {
            if (t / nbt != row) {
                row = t / nbt;
                large = ma[row * kRows + (warp & 3) * 32 + lane].large;
                all_a = shared_marks(large);
            }
            const unsigned long long mine_b = ahead;
            if (t + 1 < t1) ahead = large_b(t + 1);
            if (!(all_a & shared_marks(mine_b))) {
#pragma unroll
                for (int j = 0; j < kJoinCols; j++) rest |= (large & __shfl_sync(~0u, mine_b, j) ? 0u : 1u) << j;
                if (rest) {  // (of those, outputs whose products are all 0 are 0)
                    const Marks* m = mb + (t % nbt) * kCols + r0;
                    const unsigned long long some = ma[row * kRows + (warp & 3) * 32 + lane].some;
                    for (int j = 0; j < kJoinCols; j++)
                        if (!(some & m[j].some)) rest &= ~(1u << j);
                }
            }
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
            uint32_t z[kLevels][kJoinCols];
#pragma unroll
            for (int l = 0; l < kLevels; l++)
                ldN<kJoinCols>(tmem + b * kAccStep + l * kCols + r0 + ((uint32_t)(warp & 3) << 21), z[l]);
            ld_wait();
            fence_before();
            const int xa_exp = ea[xa] - kUnit - n_cuts;
#pragma unroll
            for (int j = 0; j < kJoinCols; j++) {
                auto level = [&](int l) { return __uint_as_float(z[l][j]); };
                int v[kLevels - 1];
#pragma unroll
                for (int l = 0; l < kLevels - 2; l++) v[l] = __float2int_rn(level(l));
                v[kLevels - 2] = __float2int_rn(fmaf(level(7), 0x1p-12f, level(6) * 0x1p-4f));  // to the unit
                const long long sum = ((long long)(v[0] * 256 + v[1]) << 36) + ((long long)(v[2] * 256 + v[3]) << 20) +
                                      ((long long)(v[4] * 256 + v[5]) << 4) + v[6];
                out[(xb0 + j) * na + xa] = scaled(sum, xa_exp + eb[xb0 + j]);
            }
            if (__any_sync(~0u, rest != 0)) by_pairs(U, D, ncode, na, nb, xa, xb0, rest, xa_exp + kUnit, eb, out);
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
    return 256 + align256(4 * na) + align256(4 * nb) + align256(sizeof(Marks) * na) + align256(sizeof(Marks) * nb) +
           align256(na / kRows * bytes_a(kp)) + align256(nb / kCols * bytes_b(kp));
}

cudaError_t launch_combine_tc(double* U, double* D, int n_cuts, uint64_t na, uint64_t nb, double* out,
                              void* scratch, int sms, cudaStream_t s) {
    const int ncode = 1 << (2 * n_cuts), kp = padded(ncode);
    auto* fault = (int*)scratch;
    unsigned char* p = (unsigned char*)scratch + 256;
    auto* ea = (int*)p;
    p += align256(4 * na);
    auto* eb = (int*)p;
    p += align256(4 * nb);
    auto* ma = (Marks*)p;
    p += align256(sizeof(Marks) * na);
    auto* mb = (Marks*)p;
    p += align256(sizeof(Marks) * nb);
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
    k_digit_planes<<<(unsigned)(na / 32 + nb / 32), 256, 0, s>>>(U, D, ncode, na, nb, pa, pb, ea, eb, ma, mb);
    const uint64_t tiles = (na / kRows) * (nb / kCols);
    k_combine_tc<<<(unsigned)std::min<uint64_t>(tiles, (uint64_t)sms), kThreads, smem, s>>>(
        pa, pb, ea, eb, ma, mb, (const float2*)U, (const float2*)D, n_cuts, na, nb, out, fault);
    return cudaGetLastError();
}

}  // namespace svk
