// CutQC reconstruction on the GPU (Sec. III-A, Eqs. 3.2-3.7; the Builder of
// Sec. IV-A, including its partial reconstruction over chosen qubits).
//
// Each of the K cut wires contributes one of four terms i_j in {1,2,3,4}:
//   upstream (measured variant m, outcome y of the cut qubit):
//     1: I/Z variant, weight 2 for y = 0     2: I/Z variant, weight 2 for y = 1
//     3: X variant, weight (-1)^y            4: Y variant, weight (-1)^y
//   downstream (initialisation s of the cut qubit):
//     1: |0>    2: |1>    3: 2|+> - |0> - |1>    4: 2|+i> - |0> - |1>
// p(x_A, x_B) = 2^-K sum_{i in {1..4}^K} U_i(x_A) D_i(x_B).
//
// Three steps (none with atomics on float64; the marginals' partial sums are integers):
//  1. k_marginal_sweep, k_marginal_bins: every variant's distribution summed over the qubits
//     that are neither kept nor cut, exactly in 128-bit fixed point (units of
//     2^-112; a bin of a distribution is at most 1) -- the one pass over all
//     variant data;
//  2. k_up_terms / k_down_terms: U_i and D_i as exact integer combinations
//     (weights 0, +-1, +-2 per cut) of those small marginals, in signed
//     128-bit fixed point (|U| <= 2^K, |D| <= 4^K), rounded once to float64;
//  3. the [2^kb x 4^K] x [4^K x 2^ka] contraction: up to three cuts and from
//     2^20 outputs on as exact digit products on the tensor cores
//     (cut_combine.cu), else k_combine: float pairs (hi, lo: 48 significant
//     bits) tiled through shared memory, in compensated arithmetic on the FP32
//     units (error-free TwoProd and TwoSum, Ogita, Rump and Oishi 2005): absolute
//     error about 2^-47 sum_i |U_i D_i| 2^-K per output.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include "float_pair.cuh"
#include "kernels.cuh"
#include "sv.h"

namespace {

using svk::dot2_add;
using svk::pair_of;

constexpr int kMaxCuts = 6;
constexpr int kScale = 112;  // fixed-point unit 2^-112

struct CutGeom {
    int32_t K, width_a, width_b, keep_a_n, keep_b_n;
    int8_t cut_pos[kMaxCuts];   // cut qubit j inside the upstream circuit
    int8_t mq_a[40];            // upstream marginal qubits in bin-bit order (kept ascending, then cut j)
    int8_t mq_b[40];            // downstream kept qubits, ascending
};

__device__ __forceinline__ unsigned __int128 fixed_of(double x) {  // x >= 0
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return 0;
    const unsigned long long mant = (b & ((1ull << 52) - 1)) | (1ull << 52);
    const int sh = e - 1075 + kScale;
    if (sh >= 0) return (unsigned __int128)mant << sh;
    if (sh <= -53) return 0;
    return (unsigned __int128)(mant >> (-sh));
}

__device__ __forceinline__ double s128_to_double(unsigned __int128 v) {
    const bool neg = (unsigned long long)(v >> 64) >> 63;
    if (neg) v = ~v + 1;  // magnitude
    if (v == 0) return 0.0;
    const unsigned long long h = (unsigned long long)(v >> 64), l = (unsigned long long)v;
    const int lz = h ? __clzll(h) : 64 + __clzll(l);
    const unsigned __int128 nv = v << lz;
    unsigned long long top = (unsigned long long)(nv >> 64);
    top |= ((unsigned long long)nv != 0ull) ? 1ull : 0ull;
    const double d = ldexp(__ull2double_rn(top), 64 - lz - kScale);
    return neg ? -d : d;
}

__device__ __forceinline__ unsigned __int128 ld128(const unsigned long long* p, uint64_t i) {
    return ((unsigned __int128)p[2 * i + 1] << 64) | p[2 * i];
}
// lo, hi += x in units of 2^-112.  Below 2^-60 x takes the general form; up to
// 1, which is all a distribution holds, its 53 bits are shifted by at most 60.
__device__ __forceinline__ void fixed_add(unsigned long long& lo, unsigned long long& hi, double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int sh = (int)((b >> 52) & 0x7ff) - 1075 + kScale;
    unsigned long long l, h;
    if ((unsigned)sh < 64u) {
        const unsigned long long mant = (b & ((1ull << 52) - 1)) | (1ull << 52);
        l = mant << sh;
        h = (mant >> 1) >> (63 - sh);
    } else {
        const unsigned __int128 v = fixed_of(x);
        l = (unsigned long long)v;
        h = (unsigned long long)(v >> 64);
    }
    lo += l;
    hi += h + (lo < l ? 1 : 0);
}

// Step 1: out[v * nbins + b] = sum of p_v[i] over every i whose bits at the
// marginal qubits mq[0..nm) are b.
//
// A warp sweeps rows of 64 consecutive values (two a lane, 512 bytes): the
// marginal qubits above bit 5 choose the warp's task, the others above it the
// rows, each lane adds its two columns over the rows, and the columns that
// differ in summed qubits only are added at the end by shuffles.  Where that
// leaves too few tasks the highest summed qubits divide the rows among `parts`
// warps, which add to their bins by 64-bit integer atomics with the carry (exact
// in any order).  A warp issues the loads of eight rows before it adds the first.
// Bound by the integer pipe (90 % busy) and HBM together: 2.6 GB (27 variants of 21
// qubits with 15 marginal ones, 64 of 22 with 12) in 435 us, 6.0 TB/s, where one thread a bin with loads strided by the
// summed qubits took 713; with one row in flight 630, and with three-word sums
// on the multipliers, of fewer integer instructions, 465.
struct Sweep {
    int32_t tasks_log2, parts_log2;
    uint64_t task_mask;           // index bits of the task: marginal qubits from bit 6 on
    uint64_t part_mask, row_mask; // summed qubits from bit 6 on: chosen by the part, walked by the warp
    int8_t bin_of[40];            // bin bit of each qubit, or -1
};

__device__ __forceinline__ uint64_t deposit(uint64_t v, uint64_t mask) {
    uint64_t r = 0;
    for (; mask; mask &= mask - 1, v >>= 1)
        if (v & 1) r |= mask & (0 - mask);
    return r;
}

__global__ void __launch_bounds__(256) k_marginal_sweep(const double* const* __restrict__ var, int nvar, int nm,
                                                        const __grid_constant__ Sweep S,
                                                        unsigned long long* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = (uint64_t)gridDim.x * 8, tasks = (uint64_t)nvar << (S.tasks_log2 + S.parts_log2);
    for (uint64_t w = (uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5); w < tasks; w += warps) {
        const uint64_t part = w & ((1ull << S.parts_log2) - 1), task = (w >> S.parts_log2) & ((1ull << S.tasks_log2) - 1);
        const uint64_t v = w >> (S.parts_log2 + S.tasks_log2);
        const uint64_t high = deposit(task, S.task_mask);
        const double* p = var[v] + (high | deposit(part, S.part_mask)) + 2 * lane;
        const bool vec = ((uintptr_t)p & 15) == 0;
        unsigned long long lo[2] = {0, 0}, hi[2] = {0, 0};
        uint64_t r = 0;
        const uint64_t rows = 1ull << __popcll(S.row_mask);
        auto next = [&](double2& x) {
            if (vec) x = __ldcs(reinterpret_cast<const double2*>(p + r));
            else x = make_double2(p[r], p[r + 1]);
            r = ((r | ~S.row_mask) + 1) & S.row_mask;
        };
        constexpr int kBatch = 8;  // rows in flight: their loads are issued before the first is added
        uint64_t k = 0;
        for (; k + kBatch <= rows; k += kBatch) {
            double2 x[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; u++) next(x[u]);
#pragma unroll
            for (int u = 0; u < kBatch; u++) {
                fixed_add(lo[0], hi[0], x[u].x);
                fixed_add(lo[1], hi[1], x[u].y);
            }
        }
        for (; k < rows; k++) {
            double2 x;
            next(x);
            fixed_add(lo[0], hi[0], x.x);
            fixed_add(lo[1], hi[1], x.y);
        }
        auto add = [](unsigned long long& l, unsigned long long& h, unsigned long long l2, unsigned long long h2) {
            l += l2;
            h += h2 + (l < l2 ? 1 : 0);
        };
        if (S.bin_of[0] < 0) add(lo[0], hi[0], lo[1], hi[1]);
        bool mine = true;
        uint64_t bin = 0;
        for (int q = 1; q < 6; q++) {
            const int bit = 1 << (q - 1);
            if (S.bin_of[q] < 0) {
                for (int e = 0; e < 2; e++) {
                    const unsigned long long l = __shfl_xor_sync(~0u, lo[e], bit), h = __shfl_xor_sync(~0u, hi[e], bit);
                    add(lo[e], hi[e], l, h);
                }
                mine = mine && !(lane & bit);
            } else if (lane & bit) {
                bin |= 1ull << S.bin_of[q];
            }
        }
        for (uint64_t left = high; left; left &= left - 1) bin |= 1ull << S.bin_of[__ffsll(left) - 1];
        if (!mine) continue;
        for (int e = 0; e < (S.bin_of[0] < 0 ? 1 : 2); e++) {
            unsigned long long* o = out + 2 * ((v << nm) + (bin | (e ? 1ull << S.bin_of[0] : 0)));
            if (S.parts_log2 == 0) {
                o[0] = lo[e];
                o[1] = hi[e];
            } else {
                const unsigned long long old = atomicAdd(o, lo[e]);
                atomicAdd(o + 1, hi[e] + (old + lo[e] < old ? 1 : 0));
            }
        }
    }
}

// The same, one thread a bin: for distributions of fewer than 2^6 values, and where
// a warp of the sweep would walk fewer than 8 rows (what it does once a task then
// counts for more than the sums) and there are bins for the chip's threads.
// 27 variants of 20 qubits, three of the lowest six summed and so many above that the
// sweep has 1, 2 and 4 rows: 419 -> 95, 228 -> 73, 135 -> 71 us; with 8 rows 64 against
// the sweep's 75; with 25,000 bins the sweep is the better one (4 rows: 19 us against 35).
__global__ void k_marginal_bins(const double* const* __restrict__ var, int nvar, int width, uint64_t M,
                                 const __grid_constant__ Sweep S, int nm, unsigned long long* __restrict__ out) {
    const uint64_t total = (uint64_t)nvar << nm;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
        const uint64_t b = t & ((1ull << nm) - 1);
        const double* p = var[t >> nm];
        uint64_t base = 0;
        for (int q = 0; q < width; q++)
            if (S.bin_of[q] >= 0) base |= ((b >> S.bin_of[q]) & 1ull) << q;
        unsigned long long lo = 0, hi = 0;
        uint64_t r = 0;
        for (uint64_t k = 0; k < 1ull << (width - nm); k++) {
            fixed_add(lo, hi, p[base | r]);
            r = ((r | M) + 1) & ~M;
        }
        out[2 * t] = lo;
        out[2 * t + 1] = hi;
    }
}

// A term as the contraction takes it: a float64, or a float pair (formed here, once,
// and not by every tile that reads it: 4 cuts, 2^24 outputs, the call 3014 -> 2560 us).
__device__ __forceinline__ void put_term(double* p, double d) { *p = d; }
__device__ __forceinline__ void put_term(float2* p, double d) { *p = pair_of(d); }

// Step 2, upstream: U_code(xk) = 2^(#terms 1, 2) sum over the outcomes y of
// the cuts with terms 3, 4 of (-1)^(their y) m_v(xk, y), the other cuts' y
// fixed by the term (term 1: y = 0, term 2: y = 1).
template <typename T>
__global__ void k_up_terms(const unsigned long long* __restrict__ mup, int K, int ka, T* __restrict__ U, int ncode) {
    const uint64_t na = 1ull << ka, total = na * (uint64_t)ncode, nb_up = na << K;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
        const int code = (int)(t / na);
        const uint64_t xk = t % na;
        int v = 0, p3 = 1, shift = 0, ybase = 0, freem = 0;
        for (int j = 0; j < K; j++) {
            const int term = (code >> (2 * j)) & 3;
            v += (term <= 1 ? 0 : term - 1) * p3;
            p3 *= 3;
            if (term <= 1) {
                shift++;
                ybase |= term << j;
            } else {
                freem |= 1 << j;
            }
        }
        unsigned __int128 acc = 0;
        // every assignment of the free cuts' outcomes: subsets of freem
        int y = 0;
        for (;;) {
            const unsigned __int128 m = ld128(mup, (uint64_t)v * nb_up + xk + ((uint64_t)(ybase | y) << ka));
            if (__popc(y) & 1) acc -= m;
            else acc += m;
            if (y == freem) break;
            y = ((y | ~freem) + 1) & freem;
        }
        put_term(U + t, s128_to_double(acc << shift));
    }
}

// Step 2, downstream: D_code(xb) = sum over initialisations s of the product
// over cuts of w(term_j, s_j) m_s(xb), with w rows (1,0,0,0), (0,1,0,0),
// (-1,-1,2,0), (-1,-1,0,2).
template <typename T>
__global__ void k_down_terms(const unsigned long long* __restrict__ mdn, int K, int kb, T* __restrict__ Dn, int ncode) {
    const uint64_t nb = 1ull << kb, total = nb * (uint64_t)ncode;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
        const int code = (int)(t / nb);
        const uint64_t xb = t % nb;
        unsigned __int128 acc = 0;
        // enumerate s digit by digit: terms 1, 2 have one choice, terms 3, 4 three
        int choice[kMaxCuts], nchoice[kMaxCuts];
        for (int j = 0; j < K; j++) {
            choice[j] = 0;
            nchoice[j] = ((code >> (2 * j)) & 3) <= 1 ? 1 : 3;
        }
        for (;;) {
            int s = 0, p4 = 1, shift = 0;
            bool neg = false;
            for (int j = 0; j < K; j++) {
                const int term = (code >> (2 * j)) & 3;
                int sj;
                if (term <= 1) sj = term;
                else if (choice[j] < 2) {  // -|0>, -|1>
                    sj = choice[j];
                    neg = !neg;
                } else {  // +2 |+> (term 3) or +2 |+i> (term 4)
                    sj = term;
                    shift++;
                }
                s += sj * p4;
                p4 *= 4;
            }
            unsigned __int128 m = ld128(mdn, (uint64_t)s * nb + xb) << shift;
            if (neg) acc -= m;
            else acc += m;
            int j = 0;
            while (j < K && ++choice[j] == nchoice[j]) choice[j++] = 0;
            if (j == K) break;
        }
        put_term(Dn + t, s128_to_double(acc));
    }
}

// Step 3: out[xb na + xa] = scale sum_c U[c][xa] D[c][xb], float-pair dot
// products.  A CTA of 256 threads computes a 64 x 64 tile (4 x 4 outputs a
// thread), 32 codes at a time through shared memory.
constexpr int kTile = 64, kCodes = 32;

__global__ void __launch_bounds__(256) k_combine(const float2* __restrict__ U, const float2* __restrict__ Dn,
                                                 int ncode, uint64_t na, uint64_t nb, double scale,
                                                 double* __restrict__ out) {
    __shared__ float2 su[kCodes][kTile], sd[kCodes][kTile];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const uint64_t ta = (uint64_t)blockIdx.x * kTile;
    const uint64_t ntb = (nb + kTile - 1) / kTile;
    for (uint64_t bt = blockIdx.y; bt < ntb; bt += gridDim.y) {  // output row tiles beyond the grid's y range
    const uint64_t tb = bt * kTile;
    float s[4][4], c[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) s[i][j] = c[i][j] = 0.f;
    for (int c0 = 0; c0 < ncode; c0 += kCodes) {
        __syncthreads();
        for (int e = threadIdx.x; e < kCodes * kTile; e += 256) {
            const int cc = e / kTile, x = e % kTile;
            const bool live = c0 + cc < ncode;
            su[cc][x] = (live && ta + x < na) ? U[(uint64_t)(c0 + cc) * na + ta + x] : make_float2(0.f, 0.f);
            sd[cc][x] = (live && tb + x < nb) ? Dn[(uint64_t)(c0 + cc) * nb + tb + x] : make_float2(0.f, 0.f);
        }
        __syncthreads();
        for (int cc = 0; cc < kCodes; cc++) {
            float2 a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                a[i] = su[cc][tx + 16 * i];
                b[i] = sd[cc][ty + 16 * i];
            }
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) dot2_add(s[i][j], c[i][j], a[i], b[j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const uint64_t xa = ta + tx + 16 * i, xb = tb + ty + 16 * j;
            if (xa < na && xb < nb) out[xb * na + xa] = scale * ((double)s[i][j] + (double)c[i][j]);
        }
    }
}

unsigned grid_of(uint64_t work, int sms) {
    uint64_t g = (work + 255) / 256;
    const uint64_t cap = (uint64_t)sms * 8;
    if (g > cap) g = cap;
    return (unsigned)(g < 1 ? 1 : g);
}

// Step 1 for one side; mq: its nm marginal qubits in bin-bit order.
cudaError_t marginals(const double* const* d_var, int nvar, int width, const int8_t* mq, int nm,
                      unsigned long long* out, int sms, cudaStream_t s) {
    Sweep S;
    std::memset(&S, 0, sizeof(S));
    std::memset(S.bin_of, -1, sizeof(S.bin_of));
    uint64_t M = 0;
    for (int j = 0; j < nm; j++) {
        S.bin_of[mq[j]] = (int8_t)j;
        M |= 1ull << mq[j];
    }
    const uint64_t above = width < 6 ? 0 : ((1ull << width) - 1) & ~63ull;
    S.task_mask = M & above;
    S.row_mask = above & ~M;
    const uint64_t bins = (uint64_t)nvar << nm;
    if (width < 6 || (__builtin_popcountll(S.row_mask) < 3 && bins >= (uint64_t)sms * 192)) {
        k_marginal_bins<<<grid_of(bins, sms), 256, 0, s>>>(d_var, nvar, width, M, S, nm, out);
        return cudaGetLastError();
    }
    S.tasks_log2 = __builtin_popcountll(S.task_mask);
    // 32 warps an SM, each with 16 rows or more
    while (((uint64_t)nvar << (S.tasks_log2 + S.parts_log2)) < (uint64_t)sms * 32 &&
           __builtin_popcountll(S.row_mask) > 4) {
        const uint64_t top = 1ull << (63 - __builtin_clzll(S.row_mask));
        S.row_mask &= ~top;
        S.part_mask |= top;
        S.parts_log2++;
    }
    if (S.parts_log2) {
        const cudaError_t e = cudaMemsetAsync(out, 0, 16 * ((size_t)nvar << nm), s);
        if (e != cudaSuccess) return e;
    }
    const uint64_t warps = (uint64_t)nvar << (S.tasks_log2 + S.parts_log2);
    const uint64_t most = (uint64_t)sms * 8;  // CTAs of 8 warps: 64 warps an SM
    k_marginal_sweep<<<(unsigned)std::min((warps + 7) / 8, most), 256, 0, s>>>(d_var, nvar, nm, S, out);
    return cudaGetLastError();
}

}  // namespace

extern "C" int sv_cut_reconstruct(const double* const* up_probs, const double* const* down_probs, int n_cuts,
                                  int width_a, const int32_t* cut_pos_a, int width_b, uint64_t keep_mask_a,
                                  uint64_t keep_mask_b, double* out, size_t out_len, int out_is_device) {
    if (!up_probs || !down_probs || !cut_pos_a || !out) return SV_ERR_ARG;
    if (n_cuts < 1 || n_cuts > kMaxCuts || width_a < n_cuts + 1 || width_a > 34 || width_b < 1 || width_b > 34)
        return SV_ERR_ARG;
    CutGeom g;
    std::memset(&g, 0, sizeof(g));
    g.K = n_cuts;
    g.width_a = width_a;
    g.width_b = width_b;
    uint64_t cutmask = 0;
    for (int j = 0; j < n_cuts; j++) {
        if (cut_pos_a[j] < 0 || cut_pos_a[j] >= width_a || ((cutmask >> cut_pos_a[j]) & 1)) return SV_ERR_QUBIT;
        cutmask |= 1ull << cut_pos_a[j];
        g.cut_pos[j] = (int8_t)cut_pos_a[j];
    }
    if ((keep_mask_a & cutmask) || (keep_mask_a >> width_a) || (keep_mask_b >> width_b)) return SV_ERR_QUBIT;
    int nma = 0, nmb = 0;
    for (int q = 0; q < width_a; q++)
        if ((keep_mask_a >> q) & 1) g.mq_a[nma++] = (int8_t)q;
    g.keep_a_n = nma;
    for (int j = 0; j < n_cuts; j++) g.mq_a[nma++] = g.cut_pos[j];
    for (int q = 0; q < width_b; q++)
        if ((keep_mask_b >> q) & 1) g.mq_b[nmb++] = (int8_t)q;
    g.keep_b_n = nmb;
    if (g.keep_a_n + g.keep_b_n > 34) return SV_ERR_SIZE;
    const uint64_t na = 1ull << g.keep_a_n, nb = 1ull << g.keep_b_n;
    if (out_len != na * nb) return SV_ERR_SIZE;
    const int ncode = 1 << (2 * n_cuts);
    int nup = 1, ndown = 1;
    for (int j = 0; j < n_cuts; j++) {
        nup *= 3;
        ndown *= 4;
    }
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return SV_ERR_CUDA;
    // device scratch: pointer tables, 128-bit marginals, term tables, output
    // staging, the tensor-core contraction's operands
    const size_t ptr_bytes = (size_t)(nup + ndown) * sizeof(double*);
    const uint64_t nbin_a = na << n_cuts;
    const size_t mup_bytes = 16 * (size_t)nup * nbin_a, mdn_bytes = 16 * (size_t)ndown * nb;
    const size_t u_bytes = 8 * (size_t)ncode * na, d_bytes = 8 * (size_t)ncode * nb;
    const size_t out_bytes = out_is_device ? 0 : 8 * na * nb;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t o_mup = al(ptr_bytes), o_mdn = o_mup + al(mup_bytes),
                 o_u = o_mdn + al(mdn_bytes), o_d = o_u + al(u_bytes), o_out = o_d + al(d_bytes),
                 o_tc = o_out + al(out_bytes);
    size_t tc_bytes = svk::combine_tc_bytes(n_cuts, na, nb);  // 0: not that kernel
    unsigned char* scratch = nullptr;
    cudaError_t e = cudaMalloc(&scratch, o_tc + tc_bytes + 256);
    if (e == cudaErrorMemoryAllocation && tc_bytes) {  // k_combine does without its operands
        cudaGetLastError();
        tc_bytes = 0;
        e = cudaMalloc(&scratch, o_tc + 256);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? SV_ERR_OOM : SV_ERR_CUDA;
    }
    auto** d_ptrs = (const double**)scratch;
    auto* mup = (unsigned long long*)(scratch + o_mup);
    auto* mdn = (unsigned long long*)(scratch + o_mdn);
    double* d_out = out_is_device ? out : (double*)(scratch + o_out);
    std::vector<const double*> hp(up_probs, up_probs + nup);
    hp.insert(hp.end(), down_probs, down_probs + ndown);
    int rc = SV_OK;
    int fault = 0;  // a bounded wait of the tensor-core contraction ran out
    cudaStream_t s = nullptr;
    if (cudaMemcpy(d_ptrs, hp.data(), ptr_bytes, cudaMemcpyHostToDevice) != cudaSuccess)
        rc = SV_ERR_CUDA;
    if (rc == SV_OK) {
        if (marginals(d_ptrs, nup, width_a, g.mq_a, g.keep_a_n + n_cuts, mup, sms, s) != cudaSuccess ||
            marginals(d_ptrs + nup, ndown, width_b, g.mq_b, g.keep_b_n, mdn, sms, s) != cudaSuccess)
            rc = SV_ERR_CUDA;
        auto terms = [&](auto* U, auto* D) {
            k_up_terms<<<grid_of(na * ncode, sms), 256, 0, s>>>(mup, n_cuts, g.keep_a_n, U, ncode);
            k_down_terms<<<grid_of(nb * ncode, sms), 256, 0, s>>>(mdn, n_cuts, g.keep_b_n, D, ncode);
        };
        if (tc_bytes) {
            auto *U = (double*)(scratch + o_u), *D = (double*)(scratch + o_d);
            terms(U, D);
            if (svk::launch_combine_tc(U, D, n_cuts, na, nb, d_out, scratch + o_tc, sms, s) != cudaSuccess ||
                cudaMemcpyAsync(&fault, scratch + o_tc, sizeof(fault), cudaMemcpyDeviceToHost, s) != cudaSuccess)
                rc = SV_ERR_CUDA;
        } else {
            auto *U = (float2*)(scratch + o_u), *D = (float2*)(scratch + o_d);
            terms(U, D);
            const uint64_t gy = (nb + kTile - 1) / kTile;
            const dim3 grid((unsigned)((na + kTile - 1) / kTile), (unsigned)(gy < 65535 ? gy : 65535));
            k_combine<<<grid, 256, 0, s>>>(U, D, ncode, na, nb, 1.0 / (double)(1ull << n_cuts), d_out);
        }
        if (cudaGetLastError() != cudaSuccess) rc = SV_ERR_CUDA;
    }
    if (rc == SV_OK && !out_is_device &&
        cudaMemcpy(out, d_out, 8 * na * nb, cudaMemcpyDeviceToHost) != cudaSuccess)
        rc = SV_ERR_CUDA;
    if (rc == SV_OK && cudaDeviceSynchronize() != cudaSuccess) rc = SV_ERR_CUDA;
    if (rc == SV_OK && fault) rc = SV_ERR_TIMEOUT;
    cudaFree(scratch);
    return rc;
}
