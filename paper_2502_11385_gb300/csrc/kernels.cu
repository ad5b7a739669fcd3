// sm_103a kernels of the statevector engine.
//
//   K1 k_init          amp := e_basis
//   K5 k_tile_pass     cache-blocked pass: gather a tile of 2^m amplitudes over
//                      the pass's local qubits into shared memory, apply the
//                      pass's fused blocks in order, write the tile back
//                      (the single-GPU counterpart of Aer's chunk blocking,
//                      Sec. III-B, Fig. 4)
//   K7 k_probs         p_i = |a_i|^2 (Listing 3's probabilities())
//      k_norm_*        sum_i p_i, exact 128-bit fixed-point accumulation
//      k_marginal      marginal distribution over chosen qubits (the
//                      Builder's partial reconstruction, Sec. IV-A)
//
// Amplitudes are interleaved complex; index bit q is qubit q.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.cuh"
#include "sv.h"
#include "tile_common.cuh"

namespace svk {

// ---------------------------------------------------------------------------
// K1: initialise to a basis state.
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ int4 unit_vector16(int e);  // 16 bytes holding 1 at amplitude e, 0 elsewhere
template <>
__device__ __forceinline__ int4 unit_vector16<float>(int e) {
    const int one = __float_as_int(1.0f);
    return e == 0 ? make_int4(one, 0, 0, 0) : make_int4(0, 0, one, 0);
}
template <>
__device__ __forceinline__ int4 unit_vector16<double>(int) {
    const long long one = __double_as_longlong(1.0);
    return make_int4((int)(one & 0xffffffffll), (int)(one >> 32), 0, 0);
}

template <typename R>
__global__ void k_init(Cx<R>* __restrict__ a, uint64_t dim, uint64_t basis) {
    constexpr int PER = 16 / sizeof(Cx<R>);  // amplitudes per 16-byte store; dim is a multiple
    const uint64_t nvec = dim / PER;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < nvec; v += stride) {
        const int4 z = (basis / PER == v) ? unit_vector16<R>((int)(basis % PER)) : make_int4(0, 0, 0, 0);
        reinterpret_cast<int4*>(a)[v] = z;
    }
}

// ---------------------------------------------------------------------------
// K5: tile pass.
// ---------------------------------------------------------------------------
// Offset of matrix row/column b inside a group: bit j of b selects tile
// position pos[j] (pm[j] = 1 << pos[j]).
template <int K>
__device__ __forceinline__ int group_offset(int b, const int (&pm)[K]) {
    int off = 0;
#pragma unroll
    for (int j = 0; j < K; j++)
        if ((b >> j) & 1) off |= pm[j];
    return off;
}

// Groups a thread handles per step of a k-qubit dense op: each coefficient
// load then feeds G independent groups.
// (Native float64 is bound by the FP64 pipe, so it keeps one group per step.)
template <int K, typename R>
struct GroupsPerStep {
    static constexpr int value = sizeof(R) == 8 ? 1 : (K <= 2 ? 4 : (K == 3 ? 2 : 1));
};

template <int K>
__device__ __forceinline__ int insert_zero_bits(int g, const int (&pos)[K]) {
#pragma unroll
    for (int j = 0; j < K; j++) {
        const int p = pos[j];
        g = ((g >> p) << (p + 1)) | (g & ((1 << p) - 1));
    }
    return g;
}

template <int K, typename R>
__device__ __forceinline__ void op_dense(Cx<R>* sm, int m, const DevOp& op, const Cx<R>* __restrict__ M) {
    constexpr int D = 1 << K;
    constexpr int G = GroupsPerStep<K, R>::value;
    int pos[K], pm[K];
#pragma unroll
    for (int j = 0; j < K; j++) {
        pos[j] = op.pos[j];
        pm[j] = 1 << pos[j];
    }
    // the swizzle is linear over GF(2) and base / offset bits are disjoint:
    // swz(base | off) = swz(base) ^ swz(off)
    constexpr int DS = K <= 4 ? D : 1;  // 5-qubit blocks recompute offsets (registers)
    int soff[DS];
#pragma unroll
    for (int b = 0; b < DS; b++) soff[b] = swz<R>(group_offset<K>(b, pm));
    auto sofs = [&](int b) { return K <= 4 ? soff[b & (DS - 1)] : swz<R>(group_offset<K>(b, pm)); };
    const int ng = 1 << (m - K);
    for (int g0 = threadIdx.x; g0 < ng; g0 += blockDim.x * G) {
        int base[G];
        bool ok[G];
        Cx<R> a[G][D];
#pragma unroll
        for (int q = 0; q < G; q++) {
            const int g = g0 + q * blockDim.x;
            ok[q] = g < ng;
            base[q] = swz<R>(insert_zero_bits<K>(ok[q] ? g : 0, pos));
#pragma unroll
            for (int b = 0; b < D; b++) a[q][b] = sm[base[q] ^ sofs(b)];
        }
        // for blocks of up to 3 qubits the coefficient rows are
        // software-pipelined: row r + 1 is loaded while row r is multiplied
        constexpr bool kPipe = K <= 3 && sizeof(R) == 4;  // FP64 is bound by its pipe anyway
        constexpr int DP = kPipe ? D : 1;
        Cx<R> un[DP];
        if constexpr (kPipe) {
#pragma unroll
            for (int c = 0; c < D; c++) un[c] = M[c];
        }
#pragma unroll(K <= 2 ? D : 1)
        for (int r = 0; r < D; r++) {
            Cx<R> ur[DP];
            if constexpr (kPipe) {
#pragma unroll
                for (int c = 0; c < D; c++) ur[c] = un[c];
                if (r + 1 < D) {
#pragma unroll
                    for (int c = 0; c < D; c++) un[c] = M[(r + 1) * D + c];
                }
            }
            R re[G], im[G];
#pragma unroll
            for (int q = 0; q < G; q++) re[q] = im[q] = R(0);
#pragma unroll
            for (int c = 0; c < D; c++) {
                const Cx<R> u = kPipe ? ur[c % DP] : M[r * D + c];
#pragma unroll
                for (int q = 0; q < G; q++) {
                    re[q] = fmaT(u.re, a[q][c].re, re[q]);
                    re[q] = fmaT(-u.im, a[q][c].im, re[q]);
                    im[q] = fmaT(u.re, a[q][c].im, im[q]);
                    im[q] = fmaT(u.im, a[q][c].re, im[q]);
                }
            }
            const int off = sofs(r);
#pragma unroll
            for (int q = 0; q < G; q++)
                if (ok[q]) sm[base[q] ^ off] = Cx<R>{re[q], im[q]};
        }
    }
}

template <typename R, int LT = 8>  // LT = log2 of the CTA size
__device__ __forceinline__ void op_diag(Cx<R>* sm, int m, const DevOp& op, const Cx<R>* __restrict__ M,
                                        uint64_t tile_base) {
    const DiagIndex d = diag_index<R, LT>(op, tile_base, threadIdx.x);
    constexpr int U = sizeof(R) == 4 ? 4 : 2;
    if (op.flags & OPF_SIGN_ONLY)
        diag_sweep<U, LT, R>(sm, m, d, threadIdx.x, M, [](Cx<R> u, Cx<R> a) { return u.re < R(0) ? Cx<R>{-a.re, -a.im} : a; });
    else
        diag_sweep<U, LT, R>(sm, m, d, threadIdx.x, M, [](Cx<R> u, Cx<R> a) {
            return Cx<R>{fmaT(u.re, a.re, -u.im * a.im), fmaT(u.re, a.im, u.im * a.re)};
        });
}

// ---------------------------------------------------------------------------
// Permutation blocks (X, Y, CX, SWAP with diagonal gates whose phases are
// powers of i): out[r] = i^code(r) in[src(r)] inside every group of 2^k
// amplitudes, moved along the permutation's cycles with one temporary (each
// amplitude read once and written once); i^code is a swap of the real and
// imaginary parts and sign changes, exact in every tile format.  The moves
// (dst | code << 5 | end-of-cycle << 7, in cycle order) are the op's
// coefficient elements, decoded by the caller's mv(t).
// ---------------------------------------------------------------------------
// Groups of a k-qubit op: zero bits inserted at the op's tile positions.
__device__ __forceinline__ int group_base(int g, const int (&pos)[5], int k) {
#pragma unroll
    for (int j = 0; j < 5; j++)
        if (j < k) g = ((g >> pos[j]) << (pos[j] + 1)) | (g & ((1 << pos[j]) - 1));
    return g;
}

// s_mv: the op's moves in cycle order, s_src: per output row r, the row it
// takes its amplitude from and the phase code (src | code << 5); both staged
// in shared memory by the caller.  Blocks of up to 3 qubits move a group's
// 2^k amplitudes through registers (all reads, then all writes); larger
// blocks follow the cycles with one temporary.
template <int K, typename S, typename SwzT>
__device__ __forceinline__ void op_perm(S* sm, int m, const DevOp& op, const int* s_mv, const int* s_src, int tid,
                                        int nthreads, S (*rot)(S, int)) {
    constexpr int D = 1 << K;
    int sp[5], pos[5];
#pragma unroll
    for (int j = 0; j < 5; j++) {
        pos[j] = j < K ? op.pos[j] : 31;
        sp[j] = j < K ? swz<SwzT>(1 << op.pos[j]) : 0;
    }
    auto off = [&](int b) {
        int o = 0;
#pragma unroll
        for (int j = 0; j < K; j++)
            if ((b >> j) & 1) o ^= sp[j];
        return o;
    };
    const int ng = 1 << (m - K);
    for (int g = tid; g < ng; g += nthreads) {
        const int base = swz<SwzT>(group_base(g, pos, K));
        if constexpr (K <= 3) {
            S v[D];  // v[r] = the source of output row r (all reads before any write)
#pragma unroll
            for (int r = 0; r < D; r++) v[r] = sm[base ^ off(s_src[r] & 31)];
#pragma unroll
            for (int r = 0; r < D; r++) sm[base ^ off(r)] = rot(v[r], (s_src[r] >> 5) & 3);
        } else {
            for (int t = 0; t < D;) {
                int mv = s_mv[t];
                const S first = sm[base ^ off(mv & 31)];
                for (;;) {
                    const bool end = (mv & 128) != 0;
                    const int nx = end ? 0 : s_mv[t + 1];
                    const S a = end ? first : sm[base ^ off(nx & 31)];
                    sm[base ^ off(mv & 31)] = rot(a, (mv >> 5) & 3);
                    t++;
                    if (end) break;
                    mv = nx;
                }
            }
        }
    }
}

__device__ __forceinline__ Cx<float> rot_cf(Cx<float> v, int c) { return rot_i(v, c); }
__device__ __forceinline__ Cx<double> rot_cd(Cx<double> v, int c) { return rot_i(v, c); }

template <int K>
__device__ __forceinline__ void op_dense_df(DF4* sm, int m, const DevOp& op, const DF4* __restrict__ M) {
    constexpr int D = 1 << K;
    constexpr int G = K <= 3 ? 2 : 1;
    int pos[K], pm[K];
#pragma unroll
    for (int j = 0; j < K; j++) {
        pos[j] = op.pos[j];
        pm[j] = 1 << pos[j];
    }
    const int ng = 1 << (m - K);
    for (int g0 = threadIdx.x; g0 < ng; g0 += blockDim.x * G) {
        int base[G];
        bool ok[G];
        DF4 a[G][D];
#pragma unroll
        for (int q = 0; q < G; q++) {
            const int g = g0 + q * blockDim.x;
            ok[q] = g < ng;
            base[q] = swz<double>(insert_zero_bits<K>(ok[q] ? g : 0, pos));
#pragma unroll
            for (int b = 0; b < D; b++) a[q][b] = sm[base[q] ^ swz<double>(group_offset<K>(b, pm))];
        }
#pragma unroll(K <= 1 ? D : 1)
        for (int r = 0; r < D; r++) {
            const DF4* Mrow = M + r * D;
            float rh[G], rl[G], ih[G], il[G];
            {
                const DF4 u = Mrow[0];
#pragma unroll
                for (int q = 0; q < G; q++) {
                    df_mul(rh[q], rl[q], u.rh, u.rl, a[q][0].rh, a[q][0].rl);
                    df_mac(rh[q], rl[q], -u.ih, -u.il, a[q][0].ih, a[q][0].il);
                    df_mul(ih[q], il[q], u.rh, u.rl, a[q][0].ih, a[q][0].il);
                    df_mac(ih[q], il[q], u.ih, u.il, a[q][0].rh, a[q][0].rl);
                }
            }
#pragma unroll
            for (int c = 1; c < D; c++) {
                const DF4 u = Mrow[c];
#pragma unroll
                for (int q = 0; q < G; q++) {
                    df_mac(rh[q], rl[q], u.rh, u.rl, a[q][c].rh, a[q][c].rl);
                    df_mac(rh[q], rl[q], -u.ih, -u.il, a[q][c].ih, a[q][c].il);
                    df_mac(ih[q], il[q], u.rh, u.rl, a[q][c].ih, a[q][c].il);
                    df_mac(ih[q], il[q], u.ih, u.il, a[q][c].rh, a[q][c].rl);
                }
            }
            const int off = swz<double>(group_offset<K>(r, pm));
#pragma unroll
            for (int q = 0; q < G; q++) {
                df_norm(rh[q], rl[q]);
                df_norm(ih[q], il[q]);
                if (ok[q]) sm[base[q] ^ off] = DF4{rh[q], rl[q], ih[q], il[q]};
            }
        }
    }
}

__device__ __forceinline__ void op_diag_df(DF4* sm, int m, const DevOp& op, const DF4* __restrict__ M,
                                           uint64_t tile_base) {
    const DiagIndex d = diag_index<double>(op, tile_base, threadIdx.x);
    if (op.flags & OPF_SIGN_ONLY) {
        diag_sweep<2, 8, double>(sm, m, d, threadIdx.x, M, [](DF4 u, DF4 a) {
            return u.rh < 0.f ? DF4{-a.rh, -a.rl, -a.ih, -a.il} : a;
        });
    } else {
        diag_sweep<2, 8, double>(sm, m, d, threadIdx.x, M, [](DF4 u, DF4 a) {
            float rh, rl, ih, il;
            df_mul(rh, rl, u.rh, u.rl, a.rh, a.rl);
            df_mac(rh, rl, -u.ih, -u.il, a.ih, a.il);
            df_mul(ih, il, u.rh, u.rl, a.ih, a.il);
            df_mac(ih, il, u.ih, u.il, a.rh, a.rl);
            df_norm(rh, rl);
            df_norm(ih, il);
            return DF4{rh, rl, ih, il};
        });
    }
}

// ---------------------------------------------------------------------------
// K5-tc: complex128 block products on the tensor cores (exact digit split).
//
// In this mode a tile holds every amplitude component as a Q62 fixed-point
// int64 (x * 2^62; the components of a normalised state never exceed 1 in
// magnitude).  A k-qubit block (k = 3 or 4; smaller blocks are padded with
// identity qubits) y = U x is taken in real form (R = 2^(k+1) <= 32 rows and
// columns: real parts, then imaginary parts) and both operands are split into
// seven 8-bit digits, x = 2^6 sum_j X_j 2^(48 - 8j) (Q62 units; the top digit
// is signed with |X_0| <= 256, the others are bytes), likewise the matrix,
// whose digit fragments are prepared on the host.  Products of digits are
// exact in bfloat16 x bfloat16 -> float32 MMAs and the partial sums of each
// level L = i + j stay below 2^24 (at most 7 pairs x 32 terms x 2^16), so each
// level is accumulated exactly in float32.  Levels 0..6 are kept (28 digit
// pairs); y = sum_L Z_L 2^(46 - 8L) is re-assembled in int64 (the dropped
// levels contribute below 2^-50 in magnitude).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint4& a, unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// bfloat16 bits of byte k (0..3) of word w, as an exact integer in [0, 255]:
// 2^23 + b is assembled with one byte permute, then 2^23 is subtracted.
__device__ __forceinline__ unsigned bf16_byte_pair(unsigned w0, unsigned w1, unsigned sel) {
    const unsigned f0 = __byte_perm(w0, 0x4B000000u, sel);
    const unsigned f1 = __byte_perm(w1, 0x4B000000u, sel);
    const float g0 = __uint_as_float(f0) - 8388608.0f;
    const float g1 = __uint_as_float(f1) - 8388608.0f;
    return __byte_perm(__float_as_uint(g0), __float_as_uint(g1), 0x7632);  // high halves: bf16(g0) | bf16(g1) << 16
}

// Signed top digit d0 = v >> 48 of two values (|d0| <= 256), packed as bf16 x 2.
__device__ __forceinline__ unsigned bf16_top_pair(long long v0, long long v1) {
    const int d0 = (int)(v0 >> 48), d1 = (int)(v1 >> 48);
    const float g0 = __int_as_float(0x4B400000 + d0) - 12582912.0f;
    const float g1 = __int_as_float(0x4B400000 + d1) - 12582912.0f;
    return __byte_perm(__float_as_uint(g0), __float_as_uint(g1), 0x7632);
}

// Seven 8-bit digits of two Q62 values x0, x1 (v = x >> 6; digit 0 = v >> 48
// signed, digit j >= 1 = byte 6 - j of v), packed pairwise as bf16 x 2.
__device__ __forceinline__ void tc_digits_pair(long long x0, long long x1, unsigned (&out)[7]) {
    const long long v0 = x0 >> 6, v1 = x1 >> 6;
    const unsigned lo0 = (unsigned)v0, hi0 = (unsigned)((unsigned long long)v0 >> 32);
    const unsigned lo1 = (unsigned)v1, hi1 = (unsigned)((unsigned long long)v1 >> 32);
    out[0] = bf16_top_pair(v0, v1);
    out[1] = bf16_byte_pair(hi0, hi1, 0x7541);  // byte 5 of v = byte 1 of hi
    out[2] = bf16_byte_pair(hi0, hi1, 0x7540);  // byte 4 = byte 0 of hi
    out[3] = bf16_byte_pair(lo0, lo1, 0x7543);
    out[4] = bf16_byte_pair(lo0, lo1, 0x7542);
    out[5] = bf16_byte_pair(lo0, lo1, 0x7541);
    out[6] = bf16_byte_pair(lo0, lo1, 0x7540);
}

// Dense block of 3 or 4 qubits on the tensor cores (8-bit digits, levels 0..6).
// A fragments: Af[((i * MT + mt) * KT + ks) * 32 + lane] for digit i, m-tile mt,
// k-step ks.  Each warp takes n-tiles of 8 groups.  Real-form row / column k
// of a block is the real part of amplitude k (k < D) or the imaginary part of
// amplitude k - D.
template <int K>
__device__ __forceinline__ void op_dense_tc(Q2* sm, int m, const DevOp& op, const uint4* __restrict__ Af) {
    static_assert(K == 3 || K == 4, "tensor-core blocks have 3 or 4 qubits");
    constexpr int D = 1 << K, R = 2 * D, MT = R / 16, KT = R / 16;
    constexpr int ND = 7, NL = 7;
    int pos[K], pm[K];
#pragma unroll
    for (int j = 0; j < K; j++) {
        pos[j] = op.pos[j];
        pm[j] = 1 << pos[j];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int ng = 1 << (m - K), ntiles = ng >> 3;
    for (int nt = warp; nt < ntiles; nt += nwarps) {
        // B operand: this lane's column is group g of the n-tile; its rows in
        // k-step ks are ks*16 + {2t, 2t+1, 2t+8, 2t+9}.  Each amplitude it needs
        // is loaded once and both its real and imaginary digits are formed.
        const int bg = swz<double>(insert_zero_bits<K>(nt * 8 + g, pos));
        unsigned bf[KT][ND][2];
        if constexpr (K == 3) {
            // one k-step: rows 2t, 2t+1 = re of amplitudes 2t, 2t+1; rows 2t+8, 2t+9 = their im
            const Q2 a0 = sm[bg ^ swz<double>(group_offset<K>(2 * t, pm))];
            const Q2 a1 = sm[bg ^ swz<double>(group_offset<K>(2 * t + 1, pm))];
            unsigned dre[ND], dim_[ND];
            tc_digits_pair(a0.re, a1.re, dre);
            tc_digits_pair(a0.im, a1.im, dim_);
#pragma unroll
            for (int j = 0; j < ND; j++) {
                bf[0][j][0] = dre[j];
                bf[0][j][1] = dim_[j];
            }
        } else {
            // k-step 0: re of amplitudes {2t, 2t+1, 2t+8, 2t+9}; k-step 1: their im
            const Q2 a0 = sm[bg ^ swz<double>(group_offset<K>(2 * t, pm))];
            const Q2 a1 = sm[bg ^ swz<double>(group_offset<K>(2 * t + 1, pm))];
            const Q2 a2 = sm[bg ^ swz<double>(group_offset<K>(2 * t + 8, pm))];
            const Q2 a3 = sm[bg ^ swz<double>(group_offset<K>(2 * t + 9, pm))];
            unsigned d[ND];
            tc_digits_pair(a0.re, a1.re, d);
#pragma unroll
            for (int j = 0; j < ND; j++) bf[0][j][0] = d[j];
            tc_digits_pair(a2.re, a3.re, d);
#pragma unroll
            for (int j = 0; j < ND; j++) bf[0][j][1] = d[j];
            tc_digits_pair(a0.im, a1.im, d);
#pragma unroll
            for (int j = 0; j < ND; j++) bf[1][j][0] = d[j];
            tc_digits_pair(a2.im, a3.im, d);
#pragma unroll
            for (int j = 0; j < ND; j++) bf[1][j][1] = d[j];
        }
        // Every lane has built its B fragments before the first mma.sync (the
        // instruction is warp-wide), so each m-tile's outputs can be written as
        // soon as they are assembled.
        // A fragments are fetched one digit ahead so each load overlaps the
        // MMAs of the previous digit
        uint4 a_next = Af[lane];  // digit 0, m-tile 0, k-step 0
#pragma unroll 1
        for (int mt = 0; mt < MT; mt++) {
            float acc[NL][4];
#pragma unroll
            for (int L = 0; L < NL; L++) acc[L][0] = acc[L][1] = acc[L][2] = acc[L][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < KT; ks++) {
#pragma unroll
                for (int i = 0; i < ND; i++) {
                    const uint4 a = a_next;
                    // next (digit, k-step) of this m-tile, else digit 0 of the next m-tile
                    const int ni = i + 1 < ND ? i + 1 : 0;
                    const int nks = i + 1 < ND ? ks : ks + 1;
                    const int nmt = (i + 1 < ND || ks + 1 < KT) ? mt : mt + 1;
                    if (nmt < MT) a_next = Af[((ni * MT + nmt) * KT + (nks < KT ? nks : 0)) * 32 + lane];
#pragma unroll
                    for (int j = 0; j < ND; j++)
                        if (i + j < NL) mma_bf16_16816(acc[i + j], a, bf[ks][j][0], bf[ks][j][1]);
                }
            }
            __syncwarp();
#pragma unroll
            for (int e = 0; e < 4; e++) {
                // y = sum_L Z_L 2^(46 - 8L) in Q62 units = 2^6 (P01 2^32 + P23 2^16 +
                // P45) + Z_6 / 4 with P_ab = 256 Z_a + Z_b formed as 64-bit products
                // (|Z_L| <= (L+1) 2^21); two's-complement wrap of the sums is harmless
                long long z[NL];
#pragma unroll
                for (int L = 0; L < NL; L++) z[L] = __float2int_rn(acc[L][e]);
                const unsigned long long p01 = (unsigned long long)(z[0] * 256 + z[1]);
                const unsigned long long p23 = (unsigned long long)(z[2] * 256 + z[3]);
                const unsigned long long p45 = (unsigned long long)(z[4] * 256 + z[5]);
                unsigned long long v = (p01 << 32) + (p23 << 16) + p45;
                v = (v << 6) + (unsigned long long)((z[6] + 2) >> 2);
                const int row = mt * 16 + g + ((e >> 1) << 3);
                const int col = 2 * t + (e & 1);
                const int b = row & (D - 1);
                const int cg = swz<double>(insert_zero_bits<K>(nt * 8 + col, pos));
                Q2* dst = &sm[cg ^ swz<double>(group_offset<K>(b, pm))];
                if (row >> K) dst->im = (long long)v;
                else dst->re = (long long)v;
            }
        }
        __syncwarp();
    }
}

__device__ __forceinline__ void op_diag_tc(Q2* sm, int m, const DevOp& op, const Q2* __restrict__ M,
                                           uint64_t tile_base) {
    const DiagIndex d = diag_index<double>(op, tile_base, threadIdx.x);
    if (op.flags & OPF_SIGN_ONLY)
        diag_sweep<1, 8, double>(sm, m, d, threadIdx.x, M, [](Q2 u, Q2 a) { return u.re < 0 ? Q2{-a.re, -a.im} : a; });
    else
        diag_sweep<1, 8, double>(sm, m, d, threadIdx.x, M, [](Q2 u, Q2 a) {
            // three products instead of four (Gauss), each output off by less than two units
            const long long k1 = qmul(u.re, a.re + a.im);
            return Q2{k1 - qmul(a.im, u.re + u.im), k1 + qmul(a.re, u.im - u.re)};
        });
}

// ---------------------------------------------------------------------------
// K5: the tile-pass kernel, shared by the arithmetic modes.
// ---------------------------------------------------------------------------
enum TileMode { MODE_F32 = 0, MODE_F64 = 1, MODE_DF = 2, MODE_TC = 3 };
template <int MODE>
struct TileTraits;
// Bytes of one diagonal entry in a mode's coefficient array: Q62 pairs
// (tensor-core complex128), double-float quadruples, complex128 or complex64.
__host__ __device__ constexpr int diag_entry_bytes(int mode) { return mode == MODE_F32 ? 8 : 16; }
template <>
struct TileTraits<MODE_F32> {
    using Store = Cx<float>;
    using Smem = Cx<float>;
    using Coef = Cx<float>;
    using SwzT = float;
};
template <>
struct TileTraits<MODE_F64> {
    using Store = Cx<double>;
    using Smem = Cx<double>;
    using Coef = Cx<double>;
    using SwzT = double;
};
template <>
struct TileTraits<MODE_DF> {
    using Store = Cx<double>;
    using Smem = DF4;
    using Coef = DF4;
    using SwzT = double;
};
template <>
struct TileTraits<MODE_TC> {
    using Store = Cx<double>;
    using Smem = Q2;
    using Coef = uint4;  // dense: MMA fragments; diagonal: Q2 entries
    using SwzT = double;
};
// The move of a permutation op's row t, from its coefficient element.
__device__ __forceinline__ int perm_move(const Cx<float>* M, int t) { return (int)M[t].re; }
__device__ __forceinline__ int perm_move(const Cx<double>* M, int t) { return (int)M[t].re; }
__device__ __forceinline__ int perm_move(const DF4* M, int t) { return (int)M[t].rh; }
__device__ __forceinline__ int perm_move(const uint4* M, int t) { return (int)M[t].x; }
__device__ __forceinline__ Cx<float> perm_rot(Cx<float> v, int c) { return rot_cf(v, c); }
__device__ __forceinline__ Cx<double> perm_rot(Cx<double> v, int c) { return rot_cd(v, c); }
__device__ __forceinline__ DF4 perm_rot(DF4 v, int c) { return rot_df(v, c); }
__device__ __forceinline__ Q2 perm_rot(Q2 v, int c) { return rot_q(v, c); }

// Stages a permutation op's moves in shared memory (every thread of the CTA
// takes part: it holds two CTA barriers) and applies it.
template <typename S, typename SwzT, typename C>
__device__ __forceinline__ void apply_perm(S* sm, int m, const DevOp& op, const C* __restrict__ M) {
    __shared__ int s_mv[32], s_src[32];
    const int D = 1 << op.k, t = threadIdx.x;
    __syncthreads();  // the previous op's reads of the tables are done
    if (t < D) s_mv[t] = perm_move(M, t);
    __syncthreads();
    if (t < D) {  // row a_t takes its amplitude from the next row of its cycle
        const int v = s_mv[t];
        int nx;
        if (v & 128) {  // last of its cycle: from the cycle's first row
            int u = t;
            while (u > 0 && !(s_mv[u - 1] & 128)) u--;
            nx = s_mv[u];
        } else {
            nx = s_mv[t + 1];
        }
        s_src[v & 31] = (nx & 31) | (v & 0x60);
    }
    __syncthreads();
    auto rot = static_cast<S (*)(S, int)>(perm_rot);
    switch (op.k) {
        case 1: op_perm<1, S, SwzT>(sm, m, op, s_mv, s_src, t, blockDim.x, rot); break;
        case 2: op_perm<2, S, SwzT>(sm, m, op, s_mv, s_src, t, blockDim.x, rot); break;
        case 3: op_perm<3, S, SwzT>(sm, m, op, s_mv, s_src, t, blockDim.x, rot); break;
        case 4: op_perm<4, S, SwzT>(sm, m, op, s_mv, s_src, t, blockDim.x, rot); break;
        default: op_perm<5, S, SwzT>(sm, m, op, s_mv, s_src, t, blockDim.x, rot); break;
    }
}

template <int MODE, int KMAX>
__device__ __forceinline__ void apply_op(typename TileTraits<MODE>::Smem* sm, int m, const DevOp& op,
                                         const typename TileTraits<MODE>::Coef* __restrict__ M, uint64_t base) {
    if (op.kind == OP_PERM) {
        apply_perm<typename TileTraits<MODE>::Smem, typename TileTraits<MODE>::SwzT>(sm, m, op, M);
        return;
    }
    if constexpr (MODE == MODE_TC) {
        if (op.kind == OP_DIAG) {
            op_diag_tc(sm, m, op, reinterpret_cast<const Q2*>(M), base);
        } else if (op.k <= 3) {
            op_dense_tc<3>(sm, m, op, M);
        } else {
            op_dense_tc<(KMAX >= 4 ? 4 : 3)>(sm, m, op, M);  // the planner caps these blocks at 4 qubits
        }
    } else if constexpr (MODE == MODE_DF) {
        if (op.kind == OP_DIAG) {
            op_diag_df(sm, m, op, M, base);
        } else if (op.k == 1) {
            op_dense_df<1>(sm, m, op, M);
        } else if (op.k == 2) {
            op_dense_df<(KMAX >= 2 ? 2 : 1)>(sm, m, op, M);
        } else if (op.k == 3) {
            op_dense_df<(KMAX >= 3 ? 3 : 1)>(sm, m, op, M);
        } else if (op.k == 4) {
            op_dense_df<(KMAX >= 4 ? 4 : 1)>(sm, m, op, M);
        } else {
            op_dense_df<(KMAX >= 5 ? 5 : 1)>(sm, m, op, M);
        }
    } else {
        using R = typename TileTraits<MODE>::SwzT;
        if (op.kind == OP_DIAG) {
            op_diag<R>(sm, m, op, M, base);
        } else if (op.k == 1) {
            op_dense<1, R>(sm, m, op, M);
        } else if (op.k == 2) {
            op_dense<(KMAX >= 2 ? 2 : 1), R>(sm, m, op, M);
        } else if (op.k == 3) {
            op_dense<(KMAX >= 3 ? 3 : 1), R>(sm, m, op, M);
        } else if (op.k == 4) {
            op_dense<(KMAX >= 4 ? 4 : 1), R>(sm, m, op, M);
        } else {
            op_dense<(KMAX >= 5 ? 5 : 1), R>(sm, m, op, M);
        }
    }
}

// Sweeps the tiles of every (state, pass) entry: gather the tile's 2^m
// amplitudes (runs of 2^c contiguous ones, 16-byte loads) into shared memory,
// apply the pass's ops in order, scatter the tile back.  Persistent: each CTA
// strides over the flattened tile space of all entries.
template <int MODE, int KMAX>
__global__ void __launch_bounds__(kTileThreads, MODE == MODE_TC ? 2 : 1)
    k_tile_pass(const BatchEntry* __restrict__ E, int n_entries, uint64_t total_tiles, const DevOp* __restrict__ ops,
                const typename TileTraits<MODE>::Coef* __restrict__ coef) {
    using Tr = TileTraits<MODE>;
    using Store = typename Tr::Store;
    using Smem = typename Tr::Smem;
    using SwzT = typename Tr::SwzT;
    extern __shared__ __align__(1024) unsigned char smraw[];
    Smem* sm = reinterpret_cast<Smem*>(smraw);
    __shared__ uint64_t dep[2][32];  // deposit tables for the tile's high local bits
    __shared__ __align__(16) DevPass P;
    __shared__ uint64_t s_state, s_begin, s_next_base;
    constexpr int kOpCache = 48;  // the pass's op descriptors, read once per pass
    __shared__ DevOp s_ops[kOpCache];
    __shared__ __align__(16) uint4 s_diag[32];  // the current diagonal op's entries (at most 32 x 16 bytes)
    int cur = -1;
    for (uint64_t t = blockIdx.x; t < total_tiles; t += gridDim.x) {
        int lo = 0, hi = n_entries - 1;  // entry owning tile t (uniform across the CTA)
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (E[mid].tile_begin <= t) lo = mid;
            else hi = mid - 1;
        }
        if (lo != cur) {
            __syncthreads();
            const unsigned* src = reinterpret_cast<const unsigned*>(&E[lo].p);
            unsigned* dst = reinterpret_cast<unsigned*>(&P);
            for (int i = threadIdx.x; i < (int)(sizeof(DevPass) / 4); i += blockDim.x) dst[i] = src[i];
            if (threadIdx.x == 0) {
                s_state = E[lo].state;
                s_begin = E[lo].tile_begin;
            }
            __syncthreads();
            if (P.n_ops <= kOpCache) {
                const int4* osrc = reinterpret_cast<const int4*>(ops + P.op0);
                int4* odst = reinterpret_cast<int4*>(s_ops);
                for (int i = threadIdx.x; i < P.n_ops * (int)(sizeof(DevOp) / 16); i += blockDim.x) odst[i] = osrc[i];
            }
            if (threadIdx.x < 64) {
                const int w = threadIdx.x >> 5, v = threadIdx.x & 31, hb = P.m - P.c;
                uint64_t d = 0;
                for (int b = 0; b < 5; b++) {
                    const int bit = w * 5 + b;
                    if (bit < hb && ((v >> b) & 1)) d |= 1ull << P.L[P.c + bit];
                }
                dep[w][v] = d;
            }
            __syncthreads();
            cur = lo;
        }
        Store* st = reinterpret_cast<Store*>(s_state);
        const int m = P.m, c = P.c;
        const int cmask = (1 << c) - 1;
        const uint64_t tl = t - s_begin;
        uint64_t base = 0;
        for (int b = 0; b < P.n - m; b++)
            if ((tl >> b) & 1) base |= 1ull << P.NL[b];
        if (threadIdx.x == 0) {  // base of the CTA's next tile (same entry), for the L2 prefetch
            const uint64_t tn = t + gridDim.x;
            uint64_t bn = ~0ull;
            if (tn < total_tiles && tn - s_begin < P.tile_count) {
                const uint64_t tln = tn - s_begin;
                bn = 0;
                for (int b = 0; b < P.n - m; b++)
                    if ((tln >> b) & 1) bn |= 1ull << P.NL[b];
            }
            s_next_base = bn;
        }
        if constexpr (MODE == MODE_DF) {
            const int N = 1 << m;
            for (int j = threadIdx.x; j < N; j += blockDim.x) {
                const int r = j >> c;
                const uint64_t gidx = base | dep[0][r & 31] | dep[1][(r >> 5) & 31] | (uint64_t)(j & cmask);
                const Cx<double> a = st[gidx];
                DF4 v;
                d2df(a.re, v.rh, v.rl);
                d2df(a.im, v.ih, v.il);
                sm[swz<double>(j)] = v;
            }
        } else if constexpr (MODE == MODE_TC) {
            // fixed-point tile (Q62); four loads in flight per thread before the conversions
            constexpr int U = 4;
            const int N = 1 << m, nt = blockDim.x;
            for (int j0 = threadIdx.x; j0 < N; j0 += U * nt) {
                Cx<double> a[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int j = j0 + u * nt, r = j >> c;
                    if (j < N) a[u] = st[base | dep[0][r & 31] | dep[1][(r >> 5) & 31] | (uint64_t)(j & cmask)];
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int j = j0 + u * nt;
                    if (j < N) sm[swz<double>(j)] = Q2{d2q(a[u].re), d2q(a[u].im)};
                }
            }
        } else {
            constexpr int PER = 16 / sizeof(Store);  // amplitudes per 16-byte vector
            const int nvec = (1 << m) / PER, nt = blockDim.x;
            for (int v = threadIdx.x; v < nvec; v += nt) {
                const int j = v * PER, r = j >> c;
                *reinterpret_cast<int4*>(sm + swz<SwzT>(j)) = *reinterpret_cast<const int4*>(
                    st + (base | dep[0][r & 31] | dep[1][(r >> 5) & 31] | (uint64_t)(j & cmask)));
            }
        }
        __syncthreads();
        {
            // Prefetch the CTA's next tile (same entry) into L2 while this one
            // is computed: one bulk prefetch per run of 2^c contiguous
            // amplitudes (256 bytes), so the next load phase reads from L2.
            // The next tile's base comes from thread 0 (computed before the
            // load phase), so a thread adds one address and one instruction.
            const int runs = 1 << (m - c);
            const uint64_t bn = s_next_base;
            if (bn != ~0ull && (int)threadIdx.x < runs) {
                const int r = threadIdx.x;
                const Store* src = st + (bn | dep[0][r & 31] | dep[1][(r >> 5) & 31]);
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(src), "r"((int)(sizeof(Store) << c))
                             : "memory");
            }
        }
        const int n_ops = P.n_ops, op0 = P.op0;
        for (int o = 0; o < n_ops; o++) {
            const DevOp op = n_ops <= kOpCache ? s_ops[o] : ops[op0 + o];
            // a diagonal op's 2^k entries (at most 32) are staged in shared
            // memory by every thread, so each amplitude reads its phase there
            // (the previous op ended with a barrier)
            const typename Tr::Coef* opc = coef + op.coeff;
            if (op.kind == OP_DIAG) {
                constexpr int kEB = diag_entry_bytes(MODE);
                const unsigned* src = reinterpret_cast<const unsigned*>(opc);
                unsigned* dst = reinterpret_cast<unsigned*>(s_diag);
                for (int i = threadIdx.x; i < (kEB / 4) << op.k; i += blockDim.x) dst[i] = src[i];
                __syncthreads();
                opc = reinterpret_cast<const typename Tr::Coef*>(s_diag);
            }
            apply_op<MODE, KMAX>(sm, m, op, opc, base);
            __syncthreads();
        }
        if constexpr (MODE == MODE_DF) {
            const int N = 1 << m;
            for (int j = threadIdx.x; j < N; j += blockDim.x) {
                const int r = j >> c;
                const uint64_t gidx = base | dep[0][r & 31] | dep[1][(r >> 5) & 31] | (uint64_t)(j & cmask);
                const DF4 v = sm[swz<double>(j)];
                st[gidx] = Cx<double>{df2d(v.rh, v.rl), df2d(v.ih, v.il)};
            }
        } else if constexpr (MODE == MODE_TC) {
            const int N = 1 << m;
            for (int j = threadIdx.x; j < N; j += blockDim.x) {
                const int r = j >> c;
                const Q2 v = sm[swz<double>(j)];
                st[base | dep[0][r & 31] | dep[1][(r >> 5) & 31] | (uint64_t)(j & cmask)] = Cx<double>{q2d(v.re), q2d(v.im)};
            }
        } else {
            constexpr int PER = 16 / sizeof(Store);
            const int nvec = (1 << m) / PER;
            for (int v = threadIdx.x; v < nvec; v += blockDim.x) {
                const int j = v * PER;
                const int r = j >> c;
                const uint64_t dj = dep[0][r & 31] | dep[1][(r >> 5) & 31] | (uint64_t)(j & cmask);
                *reinterpret_cast<int4*>(st + (base | dj)) = *reinterpret_cast<const int4*>(sm + swz<SwzT>(j));
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// K7: probabilities, exact norm, marginals.
// ---------------------------------------------------------------------------
// |v|^2, rounded once to float64.  complex128 takes two float64 operations an
// amplitude, which the FP64 pipe (1.7 a clock and SM) does in about the time of
// the HBM sweep.  complex64 would take two conversions more (2 a clock and SM),
// three times the sweep, so its squares and their sum are formed in integers:
// both squares exact in 48 bits, the smaller one aligned under the larger with a
// sticky bit, one rounding to nearest even.  Same values; 2^28 amplitudes (4.3 GB)
// 2.01 -> 0.96 ms.  Components within 2^7 of each other, by far the most, need
// no sticky bit (the squares have 14 bits to spare) and their sum's leading bit is
// one of three: 0.96 -> 0.81 ms, 5.3 TB/s.
__device__ __forceinline__ double prob_of(Cx<double> v) { return fma(v.re, v.re, v.im * v.im); }
__device__ __forceinline__ double prob_of(Cx<float> v) {
    const unsigned x = __float_as_uint(v.re) & 0x7FFFFFFFu, y = __float_as_uint(v.im) & 0x7FFFFFFFu;
    const unsigned a = max(x, y), b = min(x, y);
    const int shift = 2 * (int)((a >> 23) - (b >> 23));
    if (b >= 0x800000u && a < 0x7F800000u && shift <= 14) {
        const unsigned ma = (a & 0x7FFFFFu) | 0x800000u, mb = (b & 0x7FFFFFu) | 0x800000u;
        // in units of 2^(2 (ea - 150) - 14): [2^60, 2^63), nothing lost by the shift
        const unsigned long long sum =
            ((unsigned long long)ma * (ma << 7) << 7) + (((unsigned long long)mb * (mb << 7) << 7) >> shift);
        const int lz = __clz((int)(sum >> 32));  // 1, 2 or 3
        const unsigned long long top = sum << (lz - 1);  // [2^62, 2^63): 53 bits and ten to round off
        const unsigned long long mant = (top + 0x1FFull + ((top >> 10) & 1ull)) >> 10;
        return __longlong_as_double((long long)(((unsigned long long)(2 * (int)(a >> 23) + 771 - lz) << 52) + mant));
    }
    if (a >= 0x7F800000u) {  // infinity or NaN
        const double re = (double)v.re, im = (double)v.im;
        return fma(re, re, im * im);
    }
    const int ea = max((int)(a >> 23), 1), eb = max((int)(b >> 23), 1);  // subnormals have the exponent of 1
    const unsigned ma = (a & 0x7FFFFFu) | (a >= 0x800000u ? 0x800000u : 0u);
    const unsigned mb = (b & 0x7FFFFFu) | (b >= 0x800000u ? 0x800000u : 0u);
    const unsigned long long q = ((unsigned long long)mb * mb) << 15;
    const int d = 2 * (ea - eb);
    const unsigned long long low = d < 64 ? q >> d : 0ull;
    const unsigned long long sticky = (d < 64 ? (low << d) != q : q != 0ull) ? 1ull : 0ull;
    const unsigned long long sum = (((unsigned long long)ma * ma) << 15) + low;  // in units of 2^(2 (ea - 150) - 15)
    if (sum == 0ull) return 0.0;
    const int lz = __clzll((long long)sum);
    const unsigned long long top = sum << lz, mant = top >> 11;
    const unsigned long long rem = ((top & 0x7FFull) << 1) | sticky;  // against half a unit: 0x800
    const unsigned long long up = rem + (mant & 1ull) > 0x800ull ? 1ull : 0ull;
    const int e = 1023 + 63 - lz + 2 * (ea - 150) - 15;
    return __longlong_as_double((long long)(((unsigned long long)(e - 1) << 52) + mant + up));
}

// x 2^-down (x >= 0, x 2^-down < 16) as an unsigned 128-bit fixed-point
// number in units of 2^-124.
__device__ __forceinline__ unsigned __int128 to_fixed(double x, int down = 0) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return 0;  // zero or subnormal (below 2^-1022): below the grid
    const unsigned long long mant = (b & ((1ull << 52) - 1)) | (1ull << 52);
    const int sh = e - 1075 + 124 - down;
    if (sh >= 0) return (unsigned __int128)mant << sh;
    if (sh <= -53) return 0;
    return (unsigned __int128)(mant >> (-sh));
}

__device__ __forceinline__ double fixed_to_double(unsigned __int128 v) {
    if (v == 0) return 0.0;
    const unsigned long long hi = (unsigned long long)(v >> 64), lo = (unsigned long long)v;
    const int lz = hi ? __clzll(hi) : 64 + __clzll(lo);
    const unsigned __int128 nv = v << lz;
    unsigned long long top = (unsigned long long)(nv >> 64);
    top |= ((unsigned long long)nv != 0ull) ? 1ull : 0ull;  // sticky bit
    return ldexp(__ull2double_rn(top), 64 - lz - 124);
}

__device__ __forceinline__ unsigned __int128 warp_sum128(unsigned __int128 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long lo = (unsigned long long)v, hi = (unsigned long long)(v >> 64);
        const unsigned long long lo2 = __shfl_down_sync(0xffffffffu, lo, o);
        const unsigned long long hi2 = __shfl_down_sync(0xffffffffu, hi, o);
        v += ((unsigned __int128)hi2 << 64) | lo2;
    }
    return v;
}

__device__ __forceinline__ unsigned __int128 block_sum128(unsigned __int128 v) {
    __shared__ unsigned long long red[2][32];
    v = warp_sum128(v);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
        red[0][w] = (unsigned long long)v;
        red[1][w] = (unsigned long long)(v >> 64);
    }
    __syncthreads();
    unsigned __int128 r = 0;
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        if (lane < nw) r = ((unsigned __int128)red[1][lane] << 64) | red[0][lane];
        r = warp_sum128(r);
    }
    return r;  // valid in thread 0
}

// acc += |v|^2 2^-down in units of 2^-124 (each term truncated there): exact
// integer sums, in any order.  complex64 squares are added as integers, without
// the FP64 pipe (norm of 2^28 amplitudes 2.02 -> 0.75 ms; ProbSum below).
__device__ __forceinline__ void add_fixed(unsigned __int128& acc, Cx<double> v, int down) {
    acc += to_fixed(prob_of(v), down);
}
__device__ __forceinline__ void add_square(unsigned __int128& acc, float v, int down) {
    const unsigned a = __float_as_uint(v) & 0x7FFFFFFFu;
    const int e = max((int)(a >> 23), 1);
    const unsigned m = (a & 0x7FFFFFu) | (a >= 0x800000u ? 0x800000u : 0u);
    const unsigned long long q = (unsigned long long)m * m;  // times 2^(2 (e - 150))
    const int sh = 2 * e - 300 + 124 - down;
    if (sh >= 0) acc += (unsigned __int128)q << (sh & 127);
    else acc += q >> min(-sh, 63);
}
__device__ __forceinline__ void add_fixed(unsigned __int128& acc, Cx<float> v, int down) {
    add_square(acc, v.re, down);
    add_square(acc, v.im, down);
}

// A sum of |v|^2 2^-down in units of 2^-124, term by term as add_fixed().
template <typename R>
struct ProbSum {
    unsigned __int128 acc = 0;
    __device__ __forceinline__ ProbSum(int, int) {}
    __device__ __forceinline__ void add(Cx<R> v, int down) { add_fixed(acc, v, down); }
    __device__ __forceinline__ void flush(int) {}
};
// complex64: a component x below 2^-h in magnitude is split by two float additions
// into integers of at most 21 bits and a sign, x = H 2^(-h - 21) + L 2^(-h - 43),
// whose products H H, H L and L L are added by wide multiply-adds into 64-bit
// integers (at most 2^42 each: up to 2^20 terms between two flushes), without
// the variable shifts of the general form.  h lies 2^4.5 above the mean square of
// a 2^n state's components; what is larger, or has bits below 2^(-h - 43), takes
// the general form, so the sum stays exact and has the same bits.  The norm of
// 2^28 amplitudes (2.1 GB) 0.75 -> 0.49 ms, 4.4 TB/s.
template <>
struct ProbSum<float> {
    unsigned __int128 acc = 0;
    long long hh = 0, hl = 0, ll = 0;
    float m1, m2, top;  // 1.5 2^23 in units of H and of L; 2^-h
    int h;
    __device__ __forceinline__ ProbSum(int n, int down) {
        h = (n + 1) / 2 - 4;
        m1 = 1.5f * exp2i(2 - h);
        m2 = 1.5f * exp2i(-20 - h);
        top = 38 - 2 * h - down >= 0 ? exp2i(-h) : 0.f;  // (L L must not lie below 2^-124)
    }
    static __device__ __forceinline__ float exp2i(int e) { return __int_as_float((e + 127) << 23); }
    __device__ __forceinline__ void add(float x, int down) {
        const float t1 = __fadd_rn(x, m1), lo = __fsub_rn(x, __fsub_rn(t1, m1));
        const float t2 = __fadd_rn(lo, m2);
        if (fabsf(x) < top && lo == __fsub_rn(t2, m2)) {
            const int H = __float_as_int(t1) - __float_as_int(m1), L = __float_as_int(t2) - __float_as_int(m2);
            hh += (long long)H * H;
            hl += (long long)H * L;
            ll += (long long)L * L;
        } else {
            add_square(acc, x, down);
        }
    }
    __device__ __forceinline__ void add(Cx<float> v, int down) {
        add(v.re, down);
        add(v.im, down);
    }
    __device__ __forceinline__ void flush(int down) {
        const int sh = 38 - 2 * h - down;
        if (top == 0.f) return;
        acc += (unsigned __int128)hh << (sh + 44);
        acc += (unsigned __int128)(__int128)hl << (sh + 23);
        acc += (unsigned __int128)ll << sh;
        hh = hl = ll = 0;
    }
};
constexpr uint64_t kFlushTerms = 1ull << 20;  // terms between two flushes

// The same sum without the split: for small states, where a thread has one vector and
// the split's constants and its flush cost more than the shifts (and three more vectors
// in flight would be zeros).  Norm of 14 qubits complex64 33.6 -> 26.4 us a call, its
// marginal of one qubit 28.0 -> 25.2; norm of 16 qubits complex128 33.9 -> 26.0.
template <typename R>
struct PlainSum {
    unsigned __int128 acc = 0;
    __device__ __forceinline__ PlainSum(int, int) {}
    __device__ __forceinline__ void add(Cx<R> v, int down) { add_fixed(acc, v, down); }
    __device__ __forceinline__ void flush(int) {}
};

// Amplitudes of one 16-byte vector.
template <typename R>
struct Vec {
    static constexpr int N = 16 / sizeof(Cx<R>);
    union {
        int4 w;
        Cx<R> v[N];
    };
    __device__ __forceinline__ void load(const Cx<R>* p) { w = *reinterpret_cast<const int4*>(p); }
};

// Probabilities of len amplitudes (even), two at a time: 16-byte loads, and a
// 16-byte store where p allows it.  t of `threads` threads.
template <typename R>
__device__ __forceinline__ void probs_of(const Cx<R>* __restrict__ a, uint64_t len, double* __restrict__ p, uint64_t t,
                                         uint64_t threads) {
    const bool wide = (reinterpret_cast<uintptr_t>(p) & 15) == 0;
    for (uint64_t i = t; i < len / 2; i += threads) {
        Cx<R> x, y;
        if constexpr (sizeof(R) == 4) {
            Vec<R> v;
            v.load(a + 2 * i);
            x = v.v[0];
            y = v.v[1];
        } else {
            x = a[2 * i];
            y = a[2 * i + 1];
        }
        const double px = prob_of(x), py = prob_of(y);
        if (wide) {
            *reinterpret_cast<double2*>(p + 2 * i) = make_double2(px, py);
        } else {
            p[2 * i] = px;
            p[2 * i + 1] = py;
        }
    }
}

template <typename R>
__global__ void k_probs(const Cx<R>* __restrict__ a, uint64_t i0, uint64_t len, double* __restrict__ p) {
    probs_of<R>(a + i0, len, p, (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, (uint64_t)gridDim.x * blockDim.x);
}

template <typename R, typename Sum, int U>  // U vectors in flight
__global__ void k_norm_partial(const Cx<R>* __restrict__ a, uint64_t dim, unsigned long long* __restrict__ part,
                               int down) {
    Sum sum(63 - __clzll(dim), down);
    constexpr int N = Vec<R>::N;
    int terms = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, vecs = dim / N;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < vecs; i += U * stride) {
        Vec<R> v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (i + u * stride < vecs) v[u].load(a + N * (i + u * stride));
            else v[u].w = make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < U; u++)
#pragma unroll
            for (int e = 0; e < N; e++) sum.add(v[u].v[e], down);
        terms += 2 * N * U;
        if (terms >= (int)kFlushTerms) {
            sum.flush(down);
            terms = 0;
        }
    }
    sum.flush(down);
    const unsigned __int128 acc = block_sum128(sum.acc);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = (unsigned long long)acc;
        part[2 * blockIdx.x + 1] = (unsigned long long)(acc >> 64);
    }
}

__global__ void k_norm_final(const unsigned long long* __restrict__ part, int nparts, double* out) {
    unsigned __int128 acc = 0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x)
        acc += ((unsigned __int128)part[2 * i + 1] << 64) | part[2 * i];
    acc = block_sum128(acc);
    if (threadIdx.x == 0) *out = fixed_to_double(acc);
}

__device__ __forceinline__ void atomic_add128(unsigned long long* bin, unsigned __int128 v) {
    const unsigned long long lo = (unsigned long long)v;
    unsigned long long hi = (unsigned long long)(v >> 64);
    const unsigned long long old = atomicAdd(bin, lo);
    if (old + lo < old) hi += 1ull;  // carry out of the low word
    if (hi) atomicAdd(bin + 1, hi);
}

// A marginal as tasks of one warp each.  The index bits, from the lowest: the
// vector bit (complex64 only), lane_bits lane bits, the high bits.  A task has
// fixed values of the masked high bits and one of 2^split parts of the values
// of the others; it sweeps that part with coalesced loads, every lane summing
// its amplitudes in a register, then sums the lanes that share a bin and
// writes (split 0) or adds the result.  So each amplitude costs a load and an
// exact 128-bit addition instead of an atomic addition (in shared memory, or in
// global memory beyond 2^11 bins): 2^28 complex64 amplitudes (2.1 GB), 10 kept
// qubits, 2.11 -> 0.54 ms (0.85 before ProbSum).
struct MarginalPlan {
    uint64_t mask;       // masked qubits
    uint64_t open;       // unmasked high bits
    uint64_t high;       // masked high bits
    uint64_t rounds;     // sweep steps of a task
    uint64_t tasks;
    int32_t lane_bits, high_bits, split, n;
};

// Deposits the bits of v, from the lowest, at the set bits of m.
__device__ __forceinline__ uint64_t deposit_bits(uint64_t v, uint64_t m) {
    uint64_t d = 0;
    for (; m && v; v >>= 1, m &= m - 1)
        if (v & 1) d |= m & (~m + 1);
    return d;
}

template <typename R, typename Sum, int U>  // U vectors in flight
__global__ void __launch_bounds__(256) k_marginal(const Cx<R>* __restrict__ a, const MarginalPlan mp,
                                                  unsigned long long* __restrict__ bins) {
    constexpr int N = Vec<R>::N, VS = N == 2 ? 1 : 0;
    const int lane = threadIdx.x & 31;
    const bool live = (lane >> mp.lane_bits) == 0;
    const bool apart = VS && (mp.mask & 1);  // the two amplitudes of a vector belong to different bins
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t t = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < mp.tasks; t += warps) {
        const uint64_t hv = t & ((1ull << mp.high_bits) - 1), part = t >> mp.high_bits;
        const uint64_t base = deposit_bits(hv, mp.high) | ((uint64_t)lane << VS);
        uint64_t x = deposit_bits(part * mp.rounds, mp.open);
        Sum sum[2] = {Sum(mp.n, 0), Sum(mp.n, 0)};
        for (uint64_t r = 0; r < mp.rounds; r += U) {
            Vec<R> v[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (live && r + u < mp.rounds) v[u].load(a + (base | x));
                else v[u].w = make_int4(0, 0, 0, 0);
                x = ((x | ~mp.open) + 1) & mp.open;  // the next value of the unmasked high bits
            }
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int e = 0; e < N; e++) sum[e].add(v[u].v[e], 0);
            if ((r + U) % (kFlushTerms / 2) == 0)
                for (int e = 0; e < N; e++) sum[e].flush(0);
        }
        for (int e = 0; e < N; e++) sum[e].flush(0);
        unsigned __int128 acc[2] = {sum[0].acc, sum[1].acc};
        if (!apart) acc[0] += acc[1];
        for (int b = 0; b < mp.lane_bits; b++) {
            if ((mp.mask >> (VS + b)) & 1) continue;
#pragma unroll
            for (int e = 0; e < 2; e++) {
                const unsigned long long lo = (unsigned long long)acc[e], hi = (unsigned long long)(acc[e] >> 64);
                acc[e] += ((unsigned __int128)__shfl_xor_sync(0xffffffffu, hi, 1 << b) << 64) |
                          __shfl_xor_sync(0xffffffffu, lo, 1 << b);
            }
        }
        // the bin: the masked low bits, then the high ones; written by the lane whose unmasked bits are 0
        uint64_t low = (uint64_t)lane << VS, bin = 0;
        int nb = 0;
        for (int b = 0; b < VS + mp.lane_bits; b++)
            if ((mp.mask >> b) & 1) bin |= ((low >> b) & 1) << nb++;
        const uint64_t own = ((1ull << (VS + mp.lane_bits)) - 1) & ~mp.mask;
        if (!live || (low & own)) continue;
        bin |= hv << nb;
        for (int e = 0; e < (apart ? 2 : 1); e++) {  // (bit 0, when masked, is the bin's bit 0)
            unsigned long long* o = bins + 2 * (bin | (uint64_t)e);
            if (mp.split) {
                atomic_add128(o, acc[e]);
            } else {
                o[0] = (unsigned long long)acc[e];
                o[1] = (unsigned long long)(acc[e] >> 64);
            }
        }
    }
}

__global__ void k_bins_to_double(const unsigned long long* __restrict__ bins, uint64_t nbins, double* out) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nbins; b += stride)
        out[b] = fixed_to_double(((unsigned __int128)bins[2 * b + 1] << 64) | bins[2 * b]);
}

// Largest |component| of a state, as the bit pattern of a non-negative
// double (such patterns order like the values): atomicMax into *out.
__global__ void k_max_abs(const double* __restrict__ a, uint64_t n, unsigned long long* out) {
    unsigned long long m = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(a[i]) & 0x7FFFFFFFFFFFFFFFull;
        m = b > m ? b : m;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_down_sync(0xffffffffu, m, o);
        m = x > m ? x : m;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

__global__ void k_zero_u64(unsigned long long* p, uint64_t n) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) p[i] = 0ull;
}

// ---------------------------------------------------------------------------
// Multi-state init and probabilities (batched form): each CTA walks the
// entries in order and grid-strides over each entry's elements.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_init_multi(const StateEntry* __restrict__ E, int n_entries) {
    constexpr int PER = 16 / sizeof(Cx<R>);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (int e = 0; e < n_entries; e++) {
        Cx<R>* a = reinterpret_cast<Cx<R>*>(E[e].state);
        const uint64_t nvec = (1ull << E[e].n) / PER;
        for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < nvec; v += stride)
            reinterpret_cast<int4*>(a)[v] = (v == 0) ? unit_vector16<R>(0) : make_int4(0, 0, 0, 0);
    }
}

// The probabilities of many states, the states' blocks one after another over the
// grid.  (With every state's first amplitudes in the first CTAs, small states followed
// one another there: 608 of 8 qubits complex64 took some 300 us of a batch's 890.)
template <typename R>
__global__ void k_probs_multi(const StateEntry* __restrict__ E, int n_entries, uint64_t blocks) {
    for (uint64_t b = blockIdx.x; b < blocks; b += gridDim.x) {
        int lo = 0, hi = n_entries - 1;  // the state owning block b
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (E[mid].first <= b) lo = mid;
            else hi = mid - 1;
        }
        const StateEntry e = E[lo];
        const uint64_t i0 = (b - e.first) * kProbsBlock, dim = 1ull << e.n;
        probs_of<R>(reinterpret_cast<const Cx<R>*>(e.state) + i0, min(dim, (uint64_t)kProbsBlock),
                    reinterpret_cast<double*>(e.probs) + i0, threadIdx.x, blockDim.x);
    }
}

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
static unsigned grid_for(uint64_t work, int threads, const DevInfo& di, int per_sm = 8) {
    uint64_t g = (work + threads - 1) / threads;
    const uint64_t cap = (uint64_t)di.sms * per_sm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (unsigned)g;
}

cudaError_t launch_init(int dt, void* amp, int n, uint64_t basis, cudaStream_t s, const DevInfo& di) {
    const uint64_t dim = 1ull << n;
    if (dt == SV_C64)
        k_init<float><<<grid_for(dim / 2, 256, di), 256, 0, s>>>((Cx<float>*)amp, dim, basis);
    else
        k_init<double><<<grid_for(dim, 256, di), 256, 0, s>>>((Cx<double>*)amp, dim, basis);
    return cudaGetLastError();
}

template <int MODE, int KMAX>
static cudaError_t tile_pass_impl(const BatchEntry* d_entries, int n_entries, uint64_t total_tiles, int max_m,
                                  const DevOp* d_ops, const void* d_coef, cudaStream_t s, const DevInfo& di) {
    using Tr = TileTraits<MODE>;
    const size_t smem = ((size_t)1 << max_m) * sizeof(typename Tr::Smem);
    static int configured_dev = -1;
    static size_t dyn_max = 0;
    if (configured_dev != di.device) {
        cudaFuncAttributes fa{};
        cudaError_t e = cudaFuncGetAttributes(&fa, k_tile_pass<MODE, KMAX>);
        if (e != cudaSuccess) return e;
        dyn_max = di.smem_optin - fa.sharedSizeBytes;  // opt-in limit minus the kernel's static shared memory
        e = cudaFuncSetAttribute(k_tile_pass<MODE, KMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn_max);
        if (e != cudaSuccess) return e;
        configured_dev = di.device;
    }
    if (smem > dyn_max) return cudaErrorInvalidValue;
    const int threads = kTileThreads;
    int per_sm = 1;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tile_pass<MODE, KMAX>, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    uint64_t grid = (uint64_t)di.sms * per_sm;
    if (grid > total_tiles) grid = total_tiles;
    k_tile_pass<MODE, KMAX><<<(unsigned)grid, threads, smem, s>>>(
        d_entries, n_entries, total_tiles, d_ops, (const typename Tr::Coef*)d_coef);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t tile_pass_mode(int kmax, const BatchEntry* d_entries, int n_entries, uint64_t total_tiles,
                                  int max_m, const DevOp* d_ops, const void* d_coef, cudaStream_t s,
                                  const DevInfo& di) {
    switch (kmax) {
        case 1: return tile_pass_impl<MODE, 1>(d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
        case 2: return tile_pass_impl<MODE, 2>(d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
        case 3: return tile_pass_impl<MODE, 3>(d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
        case 4: return tile_pass_impl<MODE, 4>(d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
        default: return tile_pass_impl<MODE, 5>(d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
    }
}

cudaError_t launch_tile_pass(int dt, int arith, const BatchEntry* d_entries, int n_entries, uint64_t total_tiles,
                             int max_m, int kmax, const DevOp* d_ops, const void* d_coef, cudaStream_t s,
                             const DevInfo& di, bool few) {
    if (n_entries <= 0 || total_tiles == 0) return cudaSuccess;
    if (arith == SV_ARITH_TC)
        return launch_tile_pass_tc(dt, d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
    if ((dt == SV_C64 || arith == SV_ARITH_DF64) && tile_pass_fp32_fits(dt, total_tiles, max_m, few, di))
        return launch_tile_pass_fp32(dt, d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
    if (dt == SV_C64)
        return tile_pass_mode<MODE_F32>(kmax, d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
    if (arith == SV_ARITH_DF64)
        return tile_pass_mode<MODE_DF>(kmax, d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
    if (arith == SV_ARITH_TC_SYNC)
        return tile_pass_mode<MODE_TC>(kmax, d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
    return tile_pass_mode<MODE_F64>(kmax, d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
}

cudaError_t launch_init_multi(int dt, const StateEntry* d_entries, int n_entries, uint64_t total_amps,
                              cudaStream_t s, const DevInfo& di) {
    if (n_entries <= 0) return cudaSuccess;
    const unsigned grid = grid_for(total_amps / 2 + 1, 256, di, 8);
    if (dt == SV_C64) k_init_multi<float><<<grid, 256, 0, s>>>(d_entries, n_entries);
    else k_init_multi<double><<<grid, 256, 0, s>>>(d_entries, n_entries);
    return cudaGetLastError();
}

cudaError_t launch_probs_multi(int dt, const StateEntry* d_entries, int n_entries, uint64_t blocks, cudaStream_t s,
                               const DevInfo& di) {
    if (n_entries <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)std::min<uint64_t>(blocks, (uint64_t)di.sms * 8);
    if (dt == SV_C64) k_probs_multi<float><<<grid, 256, 0, s>>>(d_entries, n_entries, blocks);
    else k_probs_multi<double><<<grid, 256, 0, s>>>(d_entries, n_entries, blocks);
    return cudaGetLastError();
}

cudaError_t launch_max_abs_c128(const void* amp, int n, unsigned long long* d_out, cudaStream_t s,
                               const DevInfo& di) {
    const uint64_t count = 2ull << n;  // re and im of 2^n amplitudes
    k_zero_u64<<<1, 32, 0, s>>>(d_out, 1);
    k_max_abs<<<grid_for(count, 256, di), 256, 0, s>>>((const double*)amp, count, d_out);
    return cudaGetLastError();
}

cudaError_t launch_probs(int dt, const void* amp, uint64_t i0, uint64_t len, double* p, cudaStream_t s,
                         const DevInfo& di) {
    if (dt == SV_C64)
        k_probs<float><<<grid_for(len / 2, 256, di), 256, 0, s>>>((const Cx<float>*)amp, i0, len, p);
    else
        k_probs<double><<<grid_for(len / 2, 256, di), 256, 0, s>>>((const Cx<double>*)amp, i0, len, p);
    return cudaGetLastError();
}

static constexpr int kNormThreads = 256;
size_t norm_scratch_bytes(const DevInfo& di) { return (size_t)di.sms * 8 * 2 * sizeof(unsigned long long); }

cudaError_t launch_norm(int dt, const void* amp, int n, void* d_scratch, double* d_out, cudaStream_t s,
                        const DevInfo& di, int down) {
    const uint64_t dim = 1ull << n;
    const unsigned grid = grid_for(dim / (dt == SV_C64 ? 2 : 1), kNormThreads, di, 8);
    auto* part = (unsigned long long*)d_scratch;
    const bool one = dim / (dt == SV_C64 ? 2 : 1) <= (uint64_t)grid * kNormThreads;  // vector a thread
    auto sum = [&](auto kernel, auto* a) { kernel<<<grid, kNormThreads, 0, s>>>(a, dim, part, down); };
    if (dt == SV_C64)
        sum(one ? k_norm_partial<float, PlainSum<float>, 1> : k_norm_partial<float, ProbSum<float>, 4>, (const Cx<float>*)amp);
    else
        sum(one ? k_norm_partial<double, PlainSum<double>, 1> : k_norm_partial<double, ProbSum<double>, 4>,
            (const Cx<double>*)amp);
    k_norm_final<<<1, 1024, 0, s>>>(part, (int)grid, d_out);
    return cudaGetLastError();
}

cudaError_t launch_marginal(int dt, const void* amp, int n, uint64_t qubit_mask, void* d_bins, double* d_out,
                            cudaStream_t s, const DevInfo& di) {
    const int vs = dt == SV_C64 ? 1 : 0, lanes = std::min(5, n - vs);
    MarginalPlan mp{};
    mp.mask = qubit_mask;
    mp.lane_bits = lanes;
    mp.n = n;
    const uint64_t top = ((1ull << n) - 1) & ~((1ull << (vs + lanes)) - 1);  // the high bits
    mp.high = qubit_mask & top;
    mp.open = ~qubit_mask & top;
    mp.high_bits = __builtin_popcountll(mp.high);
    const int open_bits = __builtin_popcountll(mp.open);
    // parts: enough warps to fill the chip while a task keeps 32 steps, a quarter of them while
    // it keeps 8 (2^21 amplitudes complex128, 3 kept qubits: 46 us with 8 steps, 37 with 32;
    // 2^24: 91 us with all warps, 103 with a quarter)
    int want = 0;
    while ((1 << want) < di.sms * 48) want++;
    const int steps = mp.high_bits + open_bits, tasks = std::min(want, std::max(steps - 5, std::min(steps - 3, want - 2)));
    mp.split = std::max(0, std::min(tasks - mp.high_bits, open_bits));
    // small states: one step a task, 2^10 tasks at most (they add to the bins)
    const bool one = mp.split > 0 && steps <= 10;
    if (one) mp.split = open_bits;
    mp.rounds = 1ull << (open_bits - mp.split);
    mp.tasks = 1ull << (mp.high_bits + mp.split);
    const uint64_t nbins = 1ull << __builtin_popcountll(qubit_mask);
    auto* bins = (unsigned long long*)d_bins;
    if (mp.split) k_zero_u64<<<grid_for(2 * nbins, 256, di), 256, 0, s>>>(bins, 2 * nbins);
    const unsigned grid = grid_for(mp.tasks * 32, 256, di, 8);
    auto sum = [&](auto kernel, auto* a) { kernel<<<grid, 256, 0, s>>>(a, mp, bins); };
    if (dt == SV_C64)
        sum(one ? k_marginal<float, PlainSum<float>, 1> : k_marginal<float, ProbSum<float>, 4>, (const Cx<float>*)amp);
    else
        sum(one ? k_marginal<double, PlainSum<double>, 1> : k_marginal<double, ProbSum<double>, 4>, (const Cx<double>*)amp);
    k_bins_to_double<<<grid_for(nbins, 256, di), 256, 0, s>>>(bins, nbins, d_out);
    return cudaGetLastError();
}

}  // namespace svk
