// K5-tc05: the tile pass of the tensor-memory modes (tcgen05.mma), complex128
// digit products (t05) and complex64 part products (t32).
//
// Structure of the kernel.  One CTA per SM holds a tile (2^13 complex128 or
// 2^14 complex64 amplitudes, 128 KiB) and all 512 tensor-memory columns.  A
// dense block is applied in jobs: the split of 128 rows x 16 (32) slots into
// 16-bit operands in tensor memory, the MMAs of the job's two output halves,
// and the re-assembly of each half.  Jobs form one stream, each stage with
// its own warps, so that the split of job j + 1, the MMAs of job j and the
// re-assembly of job j - 1 run at the same time:
//
//   warps 4..11   split a job into one of two operand buffers
//   warps 0, 1    issue the MMAs of even and of odd jobs, half 0 then half 1, each into
//                 its accumulator (a warp issues an MMA per 45 cycles, less often than
//                 the tensor cores take one, so two take turns)
//   warps 12..19  four warps for each half: read the accumulator into registers, free
//                 it, re-assemble and store
//   warp 2        copies the blocks' operand images (bulk copies), two ops ahead
//
// Permutation and diagonal ops, and the tile's loads and stores, are done by
// all of warps 4..19 (the workers) between two barriers.
//
// The stream crosses from one dense op to the next: the tile is split by the
// bit at one position p ("split position") and each op visits the p = 0 half
// first.  As long as p is no operand, an op's first half needs only what the
// op before stored in its first half, so nothing drains between them; p
// changes (and the stream drains) where an op acts on it, and every run of
// dense ops takes the positions that last longest.
//
// What bounds it: the workers' instruction stream (split and re-assembly) for
// 3-qubit blocks, split between it and the MMA issue for the widest blocks; the
// tensor cores are active half of a dense op's time.  Before, split, MMAs and
// re-assembly took turns in rounds with a CTA barrier each, thread 0 issued
// the MMAs (100 cycles each, its operands moving to uniform registers), and
// every wait read the timer.  Picoseconds per amplitude of a dense block, by
// sv_calibrate, before and now: complex128 5.0 (any width) -> 2.9 (3 qubits),
// 3.1 (4); complex64 3.3 -> 1.7 (3), 2.3 -> 1.6 (4), 1.95 -> 1.6 (5).  With
// every warp splitting and re-assembling in turn, the waits of each job were
// shared by four amplitudes a thread only: 4.0 ps.  The benchmark circuit (30
// qubits, complex128): 495 -> 357 ms of tile passes.
#include <cuda_runtime.h>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>

#include "kernels.cuh"
#include "sv.h"
#include "tcgen05.cuh"
#include "tile_common.cuh"

namespace svk {

namespace tc {

constexpr int kWorkers = 512;              // 8 splitting and 8 re-assembling warps, 2 each per TMEM lane quarter
constexpr int kLogWorkers = 9;
// the issuing and the copying warp, in a warpgroup of their own.  It is the first:
// schedulers prefer their oldest warp, and the issuing warp must not wait for slots
constexpr int kSpecial = 128;
constexpr int kCta = kSpecial + kWorkers;
// registers: 640 threads are launched with 96 each (61,440); the four worker
// warpgroups take 104, the fifth keeps 64: 4 x 128 x 104 + 128 x 64 = 61,440
#define SV_TC_WORKER_REGS 104
#define SV_TC_ISSUER_REGS 64
constexpr int kOps = 48;                   // ops whose descriptors and address tables are held at a time
constexpr int kSmemMin = 116 * 1024;       // one CTA per SM (it holds all 512 TMEM columns)
constexpr int kTmemCols = 512;             // the whole of an SM's tensor memory
constexpr uint32_t kAccHalf = 128;         // accumulators of the halves at columns 0 and 128
constexpr uint32_t kACol = 256;            // operand buffers at columns 256 and 384
constexpr uint32_t kABuf = 128;

__device__ int g_fault;  // set when a bounded wait ran out (read and cleared by the host)

__device__ __forceinline__ void workers_sync() { asm volatile("barrier.cta.sync 1, 512;\n" ::: "memory"); }

// Address table of an op (kTabInts entries, built once per CTA and pass).  The
// swizzled tile index is linear over XOR in the bits of (round, p, row, slot):
// the block's amplitude bits first (slot bits, filled up with group bits when
// the block has fewer qubits than the slot), seven row bits (five lane bits,
// two of the TMEM lane quarter), the bit at the split position p, the round
// bit.  kTabLane + l: index of lane l; kTabWarp + w: of a worker warp (its
// lane quarter and its upper two slot bits); kTabSlot + b: of the slot bits
// below; kTabX, kTabR: of p and of the round.
//
// The group bits go to the tile positions that the block and p leave free.  A
// warp's 16-byte accesses are served eight lanes at a time (8-byte ones
// sixteen), so the first lane bits take free positions whose swizzled bank
// bits differ: position q >= VS lands in bank bit (q - VS) mod 3 of the
// 16-byte slot.
constexpr int kTabLane = 0, kTabWarp = 32, kTabSlot = 48, kTabX = 51, kTabR = 52, kTabInts = 54;

__device__ __forceinline__ unsigned op_positions(const DevOp& op) {  // tile positions of a dense op
    unsigned block = 0;
    for (int j = 0; j < op.k; j++) block |= 1u << op.pos[j];
    return block;
}

// Swizzled index of bit t of (round, p, row, slot).
template <typename SwzT>
__device__ __forceinline__ int op_basis(const DevOp& op, int kt, int slot_bits, int m, int p, int t) {
    constexpr int VS = sizeof(SwzT) == 4 ? 1 : 0;  // log2(amplitudes per 16-byte slot)
    if (t < kt) return swz<SwzT>(1 << op.pos[t]);
    if (t == slot_bits + 7) return swz<SwzT>(1 << p);
    unsigned free_pos = ((1u << m) - 1) & ~(op_positions(op) | (1u << p));
    const int fill = slot_bits - kt;
    const int want = t < slot_bits ? 7 + (t - kt) : (t < slot_bits + 7 ? t - slot_bits : t - slot_bits - 1 + fill);
    unsigned used = 0;  // positions of the bank bits already taken
    for (int g = 0; free_pos; g++) {
        const unsigned cand = (g < 3 + VS && (free_pos & ~used)) ? free_pos & ~used : free_pos;
        const int q = __ffs((int)cand) - 1;
        if (g == want) return swz<SwzT>(1 << q);
        free_pos &= ~(1u << q);
        used |= q < VS ? 1u : 0x49249249u << (VS + (q - VS) % 3);
    }
    return 0;  // a tile smaller than the round
}

// Entry t of an op's table from its basis (16 entries).
__device__ __forceinline__ int op_entry(const uint16_t* basis, int slot_bits, int t) {
    int v = 0;
    if (t < kTabWarp) {
        for (int b = 0; b < 5; b++)
            if ((t >> b) & 1) v ^= basis[slot_bits + b];
    } else if (t < kTabSlot) {  // warp w: quarter w & 3, slot bits slot_bits - 2 (w bit 2) and slot_bits - 1 (bit 3)
        const int w = t - kTabWarp;
        if (w & 1) v ^= basis[slot_bits + 5];
        if (w & 2) v ^= basis[slot_bits + 6];
        if (w & 4) v ^= basis[slot_bits - 2];
        if (w & 8) v ^= basis[slot_bits - 1];
    } else if (t < kTabX) {
        v = basis[t - kTabSlot];
    } else {
        v = basis[slot_bits + 7 + (t - kTabX)];
    }
    return v;
}

// Split positions of the runs of dense ops: greedily, the highest position
// that stays free of operands longest.  change[o]: the stream drains before o.
__device__ __forceinline__ void plan_splits(const DevOp* ops, int n, int m, uint8_t* split, uint8_t* change) {
    int o = 0;
    while (o < n) {
        split[o] = 0;
        change[o] = 1;
        unsigned free_pos = (1u << m) - 1;
        int e = o;
        while (e < n && ops[e].kind == OP_DENSE) {
            const unsigned f = free_pos & ~op_positions(ops[e]);
            if (!f) break;
            free_pos = f;
            e++;
        }
        const int p = 31 - __clz((int)free_pos);
        for (int i = o; i < e; i++) {
            split[i] = (uint8_t)p;
            change[i] = i == o;
        }
        o = e > o ? e : o + 1;
    }
}

__device__ __forceinline__ void give_up(volatile int* dead) {
    *dead = 1;
    atomicExch(&g_fault, 1);
}

// One arrival of a warp, after its lanes' tensor-memory accesses.
__device__ __forceinline__ void warp_arrive(uint32_t mbar) {
    fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(mbar);
}

// A thread's slots of one half of a job (byte offsets in the tile).
struct Slots {
    int at;    // slot 0
    int o[3];  // slot bits (complex128: two)
};

}  // namespace tc

// ---------------------------------------------------------------------------
// K5-t05: the same digit products on the fifth-generation tensor cores
// (tcgen05.mma issued by one thread; amplitude digits and accumulators in
// tensor memory, block digits in shared memory).
//
// Here the tile holds Q56 (v = x * 2^56) in biased form,
//   u = v + kBias,  kBias = 2^56 + 0x808080808080 (mod 2^64),
// so that the bytes 0..5 of u are the balanced digits X_6..X_1 plus 128 and
// its top 16 bits are X_0 + 256: v = sum_j X_j 256^(6 - j) with |X_0| <= 256
// and X_j in [-128, 127] for j >= 1.  A digit is its byte b, zero-extended to
// 16 bits: as a float16 that is the subnormal number b 2^-24, which the tensor
// cores multiply exactly.  So one byte permute makes an operand word of two
// adjacent digits of a component, and there is nothing to subtract or to set:
// what the offsets 128 (256 for X_0) add to a level sum depends on the block
// only, and the accumulator starts at minus that.
//
// The block's digits U_j (balanced too) are held as float16 U_j 2^6, so every
// product counts units of 2^-18.  For a unitary block of up to 16 rows the
// level sums z_L = sum_{i + j = L} X_i U_j stay below 2^22 - 2^18 in magnitude,
// whatever the matrix: a row has 32 real entries with |U_j| <= 128 (j >= 1)
// and sum |U_0| <= 256 sqrt(32) + 16 (its 2-norm is 1), so |z_L| <= 256 x 4096 +
// 5 x 128 x 4096 + 128 x 1465 < 3.86e6 at L = 6, and less below.  The same bound
// holds for every partial sum (an offset digit counts X - (-128) or
// nothing yet, at most 128 U either way), so the accumulator, started at
// 1.5 * 2^23 + d_L (in units of 2^-18: near 48), holds integers below 2^24
// throughout, float32 adds them exactly in any order, and its bits are
// 0x42400000 + d_L + z_L: the level reads as an integer.
//
// A job covers 128 rows (TMEM lanes) x 16 slots: for 4-qubit blocks a row is a
// group and a slot an amplitude of it; for 3-qubit blocks the upper slot bit
// is the M-tile (256 groups a job).  Half h of a job (slot bit 3) is one MMA
// sequence into 7 x 16 accumulator columns:
//   A   (tensor memory): digits (1, 2), (3, 4), (5, 6) as three planes of one
//       column per component (two K-elements), digit 0 as a plane of two
//       components a column; component order 8 (amp >> 2) + 4 part + (amp & 3);
//   B   (shared, K-major core matrices of 8 rows x 16 bytes, no swizzle), per
//       half: for the pairs, row l 16 + r'' = (U_l, U_l-1) of the half's output
//       r'' = ((amp >> 2) & 1) 8 + part 4 + (amp & 3), l < 6; for digit 0, row
//       L 16 + r'' = U_L; and the accumulator's start, three K-elements a row;
//   D   (tensor memory, 112 fp32 columns): column L 16 + r'' = level L.
// Digit pair (i, i + 1) meets the block digits of levels i..6 in MMAs of N =
// (7 - i) 16 whose accumulator starts at column i 16: U_l of its first digit
// and U_l-1 of its second both belong to level i + l.
//
// Why halves: an accumulator of all 32 outputs (224 columns) has no room for
// a second one beside two operand buffers (112 columns each), and with one
// the MMAs wait while it is read.  Two accumulators of 112 columns alternate
// without a gap; the narrower MMAs cost 1482 tensor cycles a job instead of
// 1213 (47 at least per instruction).
// ---------------------------------------------------------------------------
namespace t05 {

using namespace tc;

// The accumulator starts every half job at its row's constant V (an integer
// near 1.5 * 2^23, in units of 2^-18): one MMA of a constant A slice (TMEM
// columns kAConst.., K-elements 2^4, 2^-7, 2^-18) by V's parts, V = v_2 2^22 +
// v_1 2^11 + v_0.
constexpr unsigned kMagicBits = 0x42400000u;  // bits of 48 = 1.5 * 2^23 units
constexpr uint32_t kAConst = 112;
constexpr unsigned kConst01 = 0x4C00u | (0x2000u << 16), kConst2 = 0x0040u;  // fp16 16, 2^-7; 2^-18
// d_3 and d_5 make the constant of the re-assembled sum vanish in its low 32
// bits; the others are 0.
constexpr int kD3 = -448, kD5 = -16256;
constexpr unsigned long long kBias = 0x0100808080808080ull;
// Byte sizes of a block image: the pairs' rows and digit 0's of one half, the starts of one half.
__host__ __device__ constexpr int halves(int k) { return k == 4 ? 2 : 1; }
__host__ __device__ constexpr int pair_bytes(int k) { return 96 * 2 * (2 << k) * 2; }
__host__ __device__ constexpr int top_bytes(int k) { return 112 * (2 << k) * 2; }
constexpr int kStartBytes = 112 * 16;
__host__ __device__ constexpr int image_bytes(int k) { return halves(k) * (pair_bytes(k) + top_bytes(k) + kStartBytes); }
constexpr int kBBytes = image_bytes(4);

// An amplitude of the tile: biased Q56 components (mod 2^64).
struct alignas(16) B2 {
    unsigned long long re, im;
};
__device__ __forceinline__ B2 rot(B2 v, int c) {  // v * i^c; -x is 2 kBias - u
    constexpr unsigned long long K2 = 2 * kBias;
    if (c == 1) return B2{K2 - v.im, v.re};
    if (c == 2) return B2{K2 - v.re, K2 - v.im};
    if (c == 3) return B2{v.im, K2 - v.re};
    return v;
}

// One output component from its seven accumulator words w_L = kMagicBits +
// d_L + z_L, biased:
//   v = sum_{L<=5} z_L 2^(8 (5 - L)) + round(z_6 / 256).
// Levels 5 and 6 meet in one float multiply-add (rounded to nearest at the
// unit, since the sum lies in [2^23, 2^24) units); level pairs P_q = 256 w_2q +
// w_2q+1 (mod 2^32) are 256 z + z' plus 0x82400000 and the d's, which does not
// wrap for |z| <= 2^22; one wide multiply-add joins them, with P_0 and P_2 the
// two words of its addend:  u = P_1 2^16 + ((P_0 + kTop) 2^32 + P_2).  d_3 and
// d_5 are chosen so that the constant is kBias in its low 32 bits; kTop
// corrects the upper ones.  Six instructions a component.
static_assert(257u * kMagicBits == 0x82400000u, "the pairs' constant keeps them from wrapping");
constexpr unsigned kPair1 = 257u * kMagicBits + (unsigned)kD3;
constexpr unsigned kPair2 = 257u * kMagicBits + (unsigned)(kD5 + 49152);  // w_6 / 256 adds 1.5 * 2^15 units
constexpr unsigned long long kJoined = (unsigned long long)kPair1 * 65536u + kPair2;
static_assert((unsigned)kJoined == (unsigned)kBias, "the pairs' constants give the low word of the bias");
constexpr unsigned kTop = (unsigned)(kBias >> 32) - (unsigned)(kJoined >> 32) - 257u * kMagicBits;
__device__ __forceinline__ unsigned long long join_levels(unsigned w0, unsigned w1, unsigned w2, unsigned w3,
                                                          unsigned w4, unsigned w5, unsigned w6) {
    const unsigned w56 = __float_as_uint(fmaf(__uint_as_float(w6), 0.00390625f, __uint_as_float(w5)));
    const unsigned p0 = w0 * 256u + (w1 + kTop), p1 = w2 * 256u + w3, p2 = w4 * 256u + w56;
    unsigned long long u;
    asm("{\n\t.reg .b64 c;\n\tmov.b64 c, {%2, %3};\n\tmad.wide.u32 %0, %1, 65536, c;\n\t}\n"
        : "=l"(u)
        : "r"(p1), "r"(p2), "r"(p0));
    return u;
}

// Splits the thread's four slots of a half job into an operand buffer: a, its
// column for them in the pairs' planes (`plane` columns each); a0, in digit 0's.
__device__ __forceinline__ void split(const unsigned char* sm, const Slots& j, bool live, uint32_t a, uint32_t a0,
                                      int plane) {
    B2 v[4];
    if (live) {
        auto ld = [&](int off) { return *reinterpret_cast<const B2*>(sm + off); };
        v[0] = ld(j.at);
        v[1] = ld(j.at ^ j.o[0]);
        v[2] = ld(j.at ^ j.o[1]);
        v[3] = ld(j.at ^ j.o[0] ^ j.o[1]);
    } else {
#pragma unroll
        for (int e = 0; e < 4; e++) v[e] = B2{0, 0};
    }
    unsigned lo[8], hi[8], d[8];  // components: re of the four, im of the four
#pragma unroll
    for (int e = 0; e < 4; e++) {
        lo[e] = (unsigned)v[e].re;
        hi[e] = (unsigned)(v[e].re >> 32);
        lo[4 + e] = (unsigned)v[e].im;
        hi[4 + e] = (unsigned)(v[e].im >> 32);
    }
#pragma unroll
    for (int e = 0; e < 8; e++) d[e] = __byte_perm(lo[e], 0u, 0x4041);  // digits 5, 6: bytes 1, 0
    st8(a + 2 * plane, d);
#pragma unroll
    for (int e = 0; e < 8; e++) d[e] = __byte_perm(lo[e], 0u, 0x4243);  // digits 3, 4: bytes 3, 2
    st8(a + plane, d);
#pragma unroll
    for (int e = 0; e < 8; e++) d[e] = __byte_perm(hi[e], 0u, 0x4041);  // digits 1, 2: bytes 5, 4
    st8(a, d);
#pragma unroll
    for (int e = 0; e < 4; e++) d[e] = __byte_perm(hi[2 * e], hi[2 * e + 1], 0x7632);  // digit 0: the top 16 bits
    st4(a0, d[0], d[1], d[2], d[3]);
}

using Words = uint32_t[7][8];
__device__ __forceinline__ void read(uint32_t acc, int level, Words& z) {
#pragma unroll
    for (int L = 0; L < 7; L++) ldN<8>(acc + L * level, z[L]);
}
__device__ __forceinline__ void store(unsigned char* sm, const Slots& j, const Words& z) {
    auto out = [&](int off, int e) {
        *reinterpret_cast<B2*>(sm + off) =
            B2{join_levels(z[0][e], z[1][e], z[2][e], z[3][e], z[4][e], z[5][e], z[6][e]),
               join_levels(z[0][e + 4], z[1][e + 4], z[2][e + 4], z[3][e + 4], z[4][e + 4], z[5][e + 4], z[6][e + 4])};
    };
    out(j.at, 0);
    out(j.at ^ j.o[0], 1);
    out(j.at ^ j.o[1], 2);
    out(j.at ^ j.o[0] ^ j.o[1], 3);
}
// Operand columns of (half h, slot bit s) in the pairs' planes and in digit 0's; columns of a plane.
__device__ __forceinline__ int a_col(int kt, int h, int s) { return kt == 4 ? 16 * h + 8 * s : 56 * h + 8 * s; }
__device__ __forceinline__ int a_top(int kt, int h, int s) { return kt == 4 ? 96 + 8 * h + 4 * s : 56 * h + 48 + 4 * s; }
__device__ __forceinline__ int a_plane(int kt) { return 2 << kt; }
__device__ __forceinline__ int acc_col(int, int s) { return 8 * s; }
__device__ __forceinline__ int acc_level(int) { return 16; }
__device__ __forceinline__ int first_row(int kt, int h, int) { return kt == 3 ? 128 * h : 0; }

// Issues half H of a job: the accumulator's start, digit 0, the pairs (1 + 7 R / 16
// MMAs).  AB: the operand buffer; b0: the image's address.
template <int K, int H, int AB>
__device__ __forceinline__ void issue(uint32_t b0) {
    constexpr int R = 2 << K, HB = K == 4 ? H : 0;  // 3-qubit blocks: the half is an M-tile, its rows of B are the same
    constexpr uint32_t d = kAccHalf * H, a = kACol + kABuf * AB + (K == 3 ? 7 * R / 2 * H : 0);
    constexpr int pairs = HB * pair_bytes(K), top = halves(K) * pair_bytes(K) + HB * top_bytes(K);
    constexpr int start = halves(K) * (pair_bytes(K) + top_bytes(K)) + HB * kStartBytes;
    const uint32_t b = b0 >> 4;
    // (K-elements 8..15 of the start's A are 0, so those of its B may repeat the first eight: lbo 0)
    mma(d, kAConst, b + desc_lo(start, 0), desc_hi(128), idesc(false, 112), false);
#pragma unroll
    for (int ks = 0; ks < R / 16; ks++)
        mma(d, a + 3 * R + ks * 8, b + desc_lo(top + ks * 256, 128), desc_hi(16 * R), idesc(false, 112), true);
#pragma unroll
    for (int q = 0; q < 3; q++)
#pragma unroll
        for (int ks = 0; ks < R / 8; ks++)
            mma(d + (1 + 2 * q) * 16, a + q * R + ks * 8, b + desc_lo(pairs + ks * 256, 128), desc_hi(32 * R),
                idesc(false, (6 - 2 * q) * 16), true);
}
template <int H, int AB>
__device__ __forceinline__ void issue_any(int kt, uint32_t b0) {
    if (kt == 3) issue<3, H, AB>(b0);
    else issue<4, H, AB>(b0);
}

// One block's image from its matrix M (D x D complex, row-major; 256 threads):
// see the layout above.  The entries are first rounded to 62 fraction bits.
__device__ void build_image(const double2* M, unsigned char* img, int k) {
    const int D = 1 << k, R = 2 * D;
    __shared__ int sums[32][7];  // per output row: the sum of U_j over its entries
    for (int i = threadIdx.x; i < 32 * 7; i += blockDim.x) sums[i / 7][i % 7] = 0;
    __syncthreads();
    auto half_bits = [](int x) { return (unsigned short)__half_as_ushort(__int2half_rn(x)); };
    unsigned char* tops = img + halves(k) * pair_bytes(k);
    for (int e = threadIdx.x; e < R * R; e += blockDim.x) {
        const int r = e / R, c = e % R, part = r / D, amp = r % D, cp = c / D, ca = c % D;
        const double2 z = M[amp * D + ca];
        const double x = part == 0 ? (cp ? -z.y : z.x) : (cp ? z.x : z.y);
        const double q = x * 4611686018427387904.0;  // 2^62
        const long long q62 = q >= 9223372036854775807.0 ? 0x7FFFFFFFFFFFFFFFll
                              : q <= -9223372036854775807.0 ? -0x7FFFFFFFFFFFFFFFll
                                                            : __double2ll_rn(q);
        const long long u = (q62 >> 6) + 0x808080808080ll;
        int d[7];
        d[0] = (int)(u >> 48);
        for (int j = 1; j < 7; j++) d[j] = (int)((u >> (8 * (6 - j))) & 255) - 128;
        const int rp = (amp >> 2) * 8 + part * 4 + (amp & 3), h = rp >> 4, row = rp & 15;
        const int comp = 8 * (ca >> 2) + 4 * cp + (ca & 3);
        for (int j = 0; j < 7; j++) {
            atomicAdd(&sums[rp][j], d[j]);
            const unsigned short v = half_bits(d[j] * 64);
            const int n = j * 16 + row;
            *(unsigned short*)(tops + h * top_bytes(k) + (n >> 3) * 16 * R + (comp >> 3) * 128 + (n & 7) * 16 + (comp & 7) * 2) = v;
            if (j == 6) continue;
            // (U_j, U_j-1): K-elements 2 comp, 2 comp + 1
            const int kq = 2 * comp;
            unsigned* w = (unsigned*)(img + h * pair_bytes(k) + (n >> 3) * 32 * R + (kq >> 3) * 128 + (n & 7) * 16 + (kq & 7) * 2);
            *w = v | ((unsigned)(j ? half_bits(d[j - 1] * 64) : 0) << 16);
        }
    }
    __syncthreads();
    unsigned char* starts = tops + halves(k) * top_bytes(k);
    for (int i = threadIdx.x; i < halves(k) * 112; i += blockDim.x) {
        const int h = i / 112, n = i % 112, L = n >> 4, rp = h * 16 + (n & 15);
        int V = 12582912 + (L == 3 ? kD3 : (L == 5 ? kD5 : 0)) - 256 * sums[rp][L];
        for (int j = 0; j < L; j++) V -= 128 * sums[rp][j];
        unsigned short* o = (unsigned short*)(starts + h * kStartBytes + n * 16);
        o[0] = half_bits(V >> 22);
        o[1] = half_bits((V >> 11) & 2047);
        o[2] = half_bits(V & 2047);
        for (int j = 3; j < 8; j++) o[j] = 0;
    }
}

// Phase u (Q62) times a biased amplitude: three products instead of four
// (Gauss): k1 = c (x + y), k2 = x (d - c), k3 = y (c + d) for u = c + i d, a =
// x + i y; re = k1 - k3, im = k1 + k2, each off by less than two units after
// the floors, as the four-product form is.  |x + y| <= sqrt(2) |a| and
// |d -/+ c| <= sqrt(2) 2^62 stay in range.
__device__ __forceinline__ B2 phase_mul(Q2 u, B2 a) {
    const long long x = (long long)(a.re - kBias), y = (long long)(a.im - kBias);
    const long long k1 = qmul(u.re, x + y);
    return B2{(unsigned long long)(k1 - qmul(y, u.re + u.im)) + kBias,
              (unsigned long long)(k1 + qmul(x, u.im - u.re)) + kBias};
}

}  // namespace t05

// ---------------------------------------------------------------------------
// K5-t32: complex64 block products on tcgen05 (bfloat16 triple split).
//
// Each float32 component x of the tile is split into three bfloat16 parts,
// x = h + m + l with h = bf16(x), m = bf16(x - h), l = bf16(x - h - m) (each
// residual is exact in float32; |x - h - m - l| <= 2^-24 |x|); the block's
// real form likewise, from its float64 entries.  The six products of parts
// (i, j) with i + j <= 2 carry float32 accuracy (the dropped ones are below
// 2^-24 relative): amplitude part i meets block parts 0..2-i in one MMA whose
// accumulator starts at level i, so level L = i + j collects in its own
// columns with float32 accumulation; the output is (Z_2 + Z_1) + Z_0.  No
// exact re-assembly is needed: complex64 only asks for float32 rounding.
//
// A job covers 128 rows x 32 slots: a slot is an amplitude of the row's group
// for 5-qubit blocks; 4- and 3-qubit blocks (smaller ones are padded to 3)
// fill the upper one or two slot bits with M-tiles.  Half h (slot bit 4) is
// one MMA sequence into 96 accumulator columns: three levels of 32 outputs
// (3-qubit blocks: two M-tiles of three levels of 16).  A (tensor memory):
// part i of the row's components, K order k' = 16 (amp >> 3) + 8 part + (amp
// & 7); B (shared, 3R x R bf16, K-major core matrices of 8 rows x 16 bytes):
// row h 96 + j 32 + r'' (5 qubits), j R + r' otherwise, r' = (amp >> 3) 16 +
// part 8 + (amp & 7).
// ---------------------------------------------------------------------------
namespace t32 {

using namespace tc;

constexpr int kBBytes = 6 * 64 * 64;  // 3R x R bf16 for R = 64

__device__ __forceinline__ unsigned bf16x2_rn(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned*>(&v);
}

// Three bfloat16 parts of two float32 values, packed pairwise (x0 low half).
__device__ __forceinline__ void bf3_pair(float x0, float x1, unsigned& h, unsigned& m, unsigned& l) {
    h = bf16x2_rn(x0, x1);
    const float r0 = x0 - __uint_as_float(h << 16), r1 = x1 - __uint_as_float(h & 0xFFFF0000u);
    m = bf16x2_rn(r0, r1);
    l = bf16x2_rn(r0 - __uint_as_float(m << 16), r1 - __uint_as_float(m & 0xFFFF0000u));
}

// Splits the thread's eight slots of a half job into the part planes of an operand
// buffer (a: its column for them, `plane` columns between parts).
__device__ __forceinline__ void split(const unsigned char* sm, const Slots& j, bool live, uint32_t a, int plane) {
    unsigned hh[8], mm[8], ll[8];  // pairs of re (0..3) and im (4..7)
    if (live) {
        Cx<float> v[8];
#pragma unroll
        for (int e = 0; e < 8; e++)
            v[e] = *reinterpret_cast<const Cx<float>*>(
                sm + (j.at ^ ((e & 1) ? j.o[0] : 0) ^ ((e & 2) ? j.o[1] : 0) ^ ((e & 4) ? j.o[2] : 0)));
#pragma unroll
        for (int e = 0; e < 4; e++) {
            bf3_pair(v[2 * e].re, v[2 * e + 1].re, hh[e], mm[e], ll[e]);
            bf3_pair(v[2 * e].im, v[2 * e + 1].im, hh[4 + e], mm[4 + e], ll[4 + e]);
        }
    } else {
#pragma unroll
        for (int e = 0; e < 8; e++) hh[e] = mm[e] = ll[e] = 0u;
    }
    st8(a, hh);
    st8(a + plane, mm);
    st8(a + 2 * plane, ll);
}

using Words = uint32_t[3][16];
__device__ __forceinline__ void read(uint32_t acc, int level, Words& z) {
#pragma unroll
    for (int L = 0; L < 3; L++) ldN<16>(acc + L * level, z[L]);
}
__device__ __forceinline__ void store(unsigned char* sm, const Slots& j, const Words& z) {
    auto y = [&](int c) { return (__uint_as_float(z[2][c]) + __uint_as_float(z[1][c])) + __uint_as_float(z[0][c]); };
#pragma unroll
    for (int e = 0; e < 8; e++)
        *reinterpret_cast<Cx<float>*>(sm + (j.at ^ ((e & 1) ? j.o[0] : 0) ^ ((e & 2) ? j.o[1] : 0) ^
                                            ((e & 4) ? j.o[2] : 0))) = Cx<float>{y(e), y(8 + e)};
}
// Operand columns of (half h, slot bit s), columns between part planes, accumulator columns.
__device__ __forceinline__ int a_col(int kt, int h, int s) {
    return kt == 5 ? 8 * (2 * h + s) : (kt == 4 ? 48 * h + 8 * s : 24 * (2 * h + s));
}
__device__ __forceinline__ int a_plane(int kt) { return 1 << kt; }
__device__ __forceinline__ int acc_col(int kt, int s) { return (kt == 3 ? 48 : 16) * s; }
__device__ __forceinline__ int acc_level(int kt) { return kt == 3 ? 16 : 32; }
__device__ __forceinline__ int first_row(int kt, int h, int s) { return kt == 5 ? 0 : (kt == 4 ? 128 * h : 128 * s + 256 * h); }

// Issues half H of a job: 3 R / 16 MMAs (3-qubit blocks: of both its M-tiles).
template <int K, int H, int AB>
__device__ __forceinline__ void issue(uint32_t b0) {
    constexpr int R = 2 << K, NT = K == 3 ? 2 : 1, N1 = K == 3 ? 16 : 32;  // M-tiles of a half, outputs per level
    constexpr uint32_t a = kACol + kABuf * AB + (K == 5 ? 0 : 48 * H);
    const uint32_t b = b0 >> 4;
#pragma unroll
    for (int t = 0; t < NT; t++)
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int ks = 0; ks < R / 16; ks++)
                mma(kAccHalf * H + 48 * t + i * N1, a + 24 * t + i * (R / 2) + ks * 8,
                    b + desc_lo((K == 5 ? 192 * R * H : 0) + ks * 256, 128), desc_hi(16 * R), idesc(true, (3 - i) * N1),
                    (i | ks) != 0);
}
template <int H, int AB>
__device__ __forceinline__ void issue_any(int kt, uint32_t b0) {
    if (kt == 3) issue<3, H, AB>(b0);
    else if (kt == 4) issue<4, H, AB>(b0);
    else issue<5, H, AB>(b0);
}

__host__ __device__ constexpr int image_bytes(int k) { return 6 * (2 << k) * (2 << k); }

// One block's image from its matrix M (D x D complex, row-major): x = h + m + l
// with h = bf16(x), m = bf16(x - h), l = bf16(x - h - m), from the float64 entry.
__device__ void build_image(const double2* M, unsigned char* img, int k) {
    const int D = 1 << k, R = 2 * D, Rh = R > 32 ? 32 : R;  // Rh: outputs of a half
    for (int e = threadIdx.x; e < R * R; e += blockDim.x) {
        const int r = e / R, c = e % R, part = r / D, amp = r % D, cp = c / D, ca = c % D;
        const double2 z = M[amp * D + ca];
        double x = part == 0 ? (cp ? -z.y : z.x) : (cp ? z.x : z.y);
        const int rp = (amp >> 3) * 16 + part * 8 + (amp & 7), kq = 16 * (ca >> 3) + 8 * cp + (ca & 7);
        for (int j = 0; j < 3; j++) {
            const __nv_bfloat16 b = __float2bfloat16_rn((float)x);
            const int n = (rp / Rh) * 3 * Rh + j * Rh + rp % Rh;
            *(__nv_bfloat16*)(img + (n >> 3) * 16 * R + (kq >> 3) * 128 + (n & 7) * 16 + (kq & 7) * 2) = b;
            x -= (double)__bfloat162float(b);
        }
    }
}

}  // namespace t32

// ---------------------------------------------------------------------------
// The kernel.
// ---------------------------------------------------------------------------
template <int N>
struct Int {
    static constexpr int value = N;
};
template <bool C64>
struct TcMode;
template <>
struct TcMode<false> {
    using Store = Cx<double>;
    using Smem = t05::B2;
    using SwzT = double;
    using DiagEntry = Q2;
    using Words = t05::Words;
    static constexpr int kSlotBits = 4, kBBytes = t05::kBBytes, kKmax = 4, VS = 0;
};
template <>
struct TcMode<true> {
    using Store = Cx<float>;
    using Smem = Cx<float>;
    using SwzT = float;
    using DiagEntry = Cx<float>;
    using Words = t32::Words;
    static constexpr int kSlotBits = 5, kBBytes = t32::kBBytes, kKmax = 5, VS = 1;
};

namespace tc {

__device__ __forceinline__ const unsigned char* image_at(const uint4* coef, int32_t offset) {
    return reinterpret_cast<const unsigned char*>(coef) + (size_t)offset * kImageUnit;
}

__device__ __forceinline__ t05::B2 turn(t05::B2 v, int c) { return t05::rot(v, c); }
__device__ __forceinline__ Cx<float> turn(Cx<float> v, int c) { return rot_i(v, c); }

// Permutation op (512 threads): out[r] = i^code(r) in[src(r)] inside every
// group of 2^K amplitudes.  Blocks of up to 3 qubits move a group through
// registers (all reads, then all writes), larger ones along the cycles.
// s_mv: dst | code << 5 | end-of-cycle << 7 in cycle order; s_src: src | code
// << 5 per output row.
template <int K, typename S, typename SwzT>
__device__ __forceinline__ void perm_groups(S* sm, int m, const DevOp& op, const int* s_mv, const int* s_src, int tid) {
    constexpr int D = 1 << K;
    int sp[K], pos[K];
#pragma unroll
    for (int j = 0; j < K; j++) {
        pos[j] = op.pos[j];
        sp[j] = swz<SwzT>(1 << pos[j]);
    }
    auto off = [&](int b) {
        int o = 0;
#pragma unroll
        for (int j = 0; j < K; j++)
            if ((b >> j) & 1) o ^= sp[j];
        return o;
    };
    const int ng = 1 << (m - K);
    for (int g = tid; g < ng; g += kWorkers) {
        int i = g;
#pragma unroll
        for (int j = 0; j < K; j++) i = ((i >> pos[j]) << (pos[j] + 1)) | (i & ((1 << pos[j]) - 1));
        const int base = swz<SwzT>(i);
        if constexpr (K <= 3) {
            S v[D];  // v[r] = the source of output row r (all reads before any write)
#pragma unroll
            for (int r = 0; r < D; r++) v[r] = sm[base ^ off(s_src[r] & 31)];
#pragma unroll
            for (int r = 0; r < D; r++) sm[base ^ off(r)] = turn(v[r], (s_src[r] >> 5) & 3);
        } else {
            for (int t = 0; t < D;) {
                int mv = s_mv[t];
                const S first = sm[base ^ off(mv & 31)];
                for (;;) {
                    const bool end = (mv & 128) != 0;
                    const int nx = end ? 0 : s_mv[t + 1];
                    const S a = end ? first : sm[base ^ off(nx & 31)];
                    sm[base ^ off(mv & 31)] = turn(a, (mv >> 5) & 3);
                    t++;
                    if (end) break;
                    mv = nx;
                }
            }
        }
    }
}

// moves: the op's coefficient words (dst | code << 5 | end-of-cycle << 7 in cycle order).
template <typename S, typename SwzT>
__device__ __forceinline__ void op_perm(S* sm, int m, const DevOp& op, const uint4* __restrict__ moves, int* s_mv,
                                        int* s_src, int t) {
    const int D = 1 << op.k;
    if (t < D) s_mv[t] = (int)moves[t].x;  // (the op before ended with a barrier)
    workers_sync();
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
    workers_sync();
    switch (op.k) {
        case 1: perm_groups<1, S, SwzT>(sm, m, op, s_mv, s_src, t); break;
        case 2: perm_groups<2, S, SwzT>(sm, m, op, s_mv, s_src, t); break;
        case 3: perm_groups<3, S, SwzT>(sm, m, op, s_mv, s_src, t); break;
        case 4: perm_groups<4, S, SwzT>(sm, m, op, s_mv, s_src, t); break;
        default: perm_groups<5, S, SwzT>(sm, m, op, s_mv, s_src, t); break;
    }
}

__device__ __forceinline__ void op_diag(t05::B2* sm, int m, const DevOp& op, const Q2* M, uint64_t base, int tid) {
    const DiagIndex d = diag_index<double, kLogWorkers>(op, base, tid);
    if (op.flags & OPF_SIGN_ONLY)
        diag_sweep<2, kLogWorkers, double>(sm, m, d, tid, M,
                                           [](Q2 u, t05::B2 a) { return u.re < 0 ? t05::rot(a, 2) : a; });
    else
        diag_sweep<1, kLogWorkers, double>(sm, m, d, tid, M, [](Q2 u, t05::B2 a) { return t05::phase_mul(u, a); });
}
__device__ __forceinline__ void op_diag(Cx<float>* sm, int m, const DevOp& op, const Cx<float>* M, uint64_t base, int tid) {
    using C = Cx<float>;
    const DiagIndex d = diag_index<float, kLogWorkers>(op, base, tid);
    if (op.flags & OPF_SIGN_ONLY)
        diag_sweep<4, kLogWorkers, float>(sm, m, d, tid, M, [](C u, C a) { return u.re < 0.f ? C{-a.re, -a.im} : a; });
    else
        diag_sweep<4, kLogWorkers, float>(sm, m, d, tid, M, [](C u, C a) {
            return C{fmaf(u.re, a.re, -u.im * a.im), fmaf(u.re, a.im, u.im * a.re)};
        });
}

}  // namespace tc

template <bool C64>
__global__ void __launch_bounds__(tc::kCta, 1)
    k_tile_pass_tc(const BatchEntry* __restrict__ E, int n_entries, uint64_t total_tiles,
                   const DevOp* __restrict__ ops, const uint4* __restrict__ coef) {
    using namespace tc;
    using Tr = TcMode<C64>;
    using Store = typename Tr::Store;
    using Smem = typename Tr::Smem;
    using SwzT = typename Tr::SwzT;
    constexpr int VS = Tr::VS, SB = Tr::kSlotBits;
    extern __shared__ __align__(1024) unsigned char smraw[];
    unsigned char* const smb = smraw + 2 * Tr::kBBytes;  // two block images, then the tile
    Smem* const sm = reinterpret_cast<Smem*>(smb);
    __shared__ __align__(16) DevPass P;
    __shared__ uint64_t s_state, s_begin;
    __shared__ __align__(8) uint64_t bars[17];
    __shared__ uint32_t s_tmem;
    __shared__ int s_dead;
    __shared__ DevOp s_ops[kOps];
    __shared__ __align__(16) uint16_t s_basis[kOps * 16], s_tab[kOps * kTabInts];
    __shared__ uint8_t s_split[kOps], s_change[kOps];
    __shared__ __align__(16) uint4 s_diag[32];  // the current diagonal op's entries
    __shared__ int s_mv[32], s_src[32];         // the current permutation
    // tile vectors of 16 bytes (kWorkers at a time): of step it, the global offset in bytes (low, high word) and the
    // swizzled tile offset in bytes
    __shared__ int4 s_step[32];
    const int tid = threadIdx.x, warp = tid >> 5;
    const uint32_t bar0 = smem_addr(bars);
    // operands of a job in buffer b written / read; accumulator h complete / read; block image in buffer b there / read
    auto ready = [&](int b) { return bar0 + 8u * b; };
    auto afree = [&](int b) { return bar0 + 8u * (2 + b); };
    auto done = [&](int h) { return bar0 + 8u * (4 + h); };
    auto accfree = [&](int h, int b) { return bar0 + 8u * (6 + 2 * b + h); };  // of jobs j = b (mod 2)
    auto bfull = [&](int b) { return bar0 + 8u * (10 + b); };
    auto bfree = [&](int b) { return bar0 + 8u * (12 + b); };
    auto stored = [&](int x) { return bar0 + 8u * (14 + x); };  // an op's half x of the tile
    const uint32_t end_bar = bar0 + 8u * 16;

    if (warp == 0) {  // warp 0 owns the tensor-memory allocation
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(&s_tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < 2; b++) {
            mbar_init(ready(b), kWorkers / 64);
            mbar_init(afree(b), 1);
            mbar_init(done(b), 1);
            mbar_init(accfree(0, b), kWorkers / 128);
            mbar_init(accfree(1, b), kWorkers / 128);
            mbar_init(bfull(b), 1);
            mbar_init(bfree(b), 2);
            mbar_init(stored(b), kWorkers / 64);
        }
        mbar_init(end_bar, 2);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        s_dead = 0;
    }
    fence_before();
    __syncthreads();
    fence_after();
    constexpr uint32_t tmem = 0;  // all 512 columns are this CTA's
    if (tid == 0 && s_tmem != tmem) give_up(&s_dead);
    if constexpr (!C64) {
        if (tid < 128) {  // the constant A slice in every TMEM lane, one lane quarter per warp
            const unsigned c[8] = {t05::kConst01, t05::kConst2, 0u, 0u, 0u, 0u, 0u, 0u};
            st8(tmem + ((uint32_t)(tid & ~31) << 16) + t05::kAConst, c);
            st_wait();
        }
    }
    fence_before();
    __syncthreads();
    fence_after();

    // ---- what every role does in the same order: entries, chunks of ops ----
    int cur = -1;
    // the entry owning tile t; loads its pass description when it changes (a barrier of the whole CTA)
    auto enter = [&](uint64_t t) {
        if (cur >= 0 && t - s_begin < P.tile_count) return false;
        int lo = cur < 0 ? 0 : cur, hi = n_entries - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (E[mid].tile_begin <= t) lo = mid;
            else hi = mid - 1;
        }
        __syncthreads();
        const unsigned* src = reinterpret_cast<const unsigned*>(&E[lo].p);
        unsigned* dst = reinterpret_cast<unsigned*>(&P);
        for (int i = tid; i < (int)(sizeof(DevPass) / 4); i += kCta) dst[i] = src[i];
        if (tid == 0) {
            s_state = E[lo].state;
            s_begin = E[lo].tile_begin;
        }
        __syncthreads();
        cur = lo;
        return true;
    };
    // global offset (amplitudes) of tile index i
    auto deposit = [&](int i) {
        uint64_t d = (uint64_t)(i & ((1 << P.c) - 1));
        for (int j = P.c; j < P.m; j++) d |= (uint64_t)((i >> j) & 1) << P.L[j];
        return d;
    };
    // the block size an op is applied with (smaller blocks are padded to 3 qubits)
    auto kt_of = [&](const DevOp& op) { return op.k <= 3 ? 3 : (op.k > Tr::kKmax ? Tr::kKmax : op.k); };
    int chunk_entry = -1, chunk_first = -1;  // what s_ops holds
    // ops [first, first + n) of the pass: descriptors, split positions, address tables
    auto load_chunk = [&](int first, int n) {
        if (chunk_entry == cur && chunk_first == first) return;
        __syncthreads();
        const int4* osrc = reinterpret_cast<const int4*>(ops + P.op0 + first);
        int4* odst = reinterpret_cast<int4*>(s_ops);
        for (int i = tid; i < n * (int)(sizeof(DevOp) / 16); i += kCta) odst[i] = osrc[i];
        if (tid < 32) {
            const int i = (tid * kWorkers) << VS;
            const uint64_t g = (i >> P.m ? 0 : deposit(i)) * sizeof(Store);
            s_step[tid] = make_int4((int)(uint32_t)g, (int)(g >> 32), swz<SwzT>(i) * (int)sizeof(Smem), 0);
        }
        __syncthreads();
        if (tid == 0) plan_splits(s_ops, n, P.m, s_split, s_change);
        __syncthreads();
        for (int i = tid; i < n * 16; i += kCta)
            s_basis[i] = s_ops[i >> 4].kind == OP_DENSE
                             ? (uint16_t)op_basis<SwzT>(s_ops[i >> 4], kt_of(s_ops[i >> 4]), SB, P.m, s_split[i >> 4], i & 15)
                             : (uint16_t)0;
        __syncthreads();
        for (int i = tid; i < n * kTabInts; i += kCta)
            s_tab[i] = (uint16_t)op_entry(s_basis + 16 * (i / kTabInts), SB, i % kTabInts);
        __syncthreads();
        chunk_entry = cur;
        chunk_first = first;
    };
    auto chunk_size = [&](int first) { return min(kOps, P.n_ops - first); };
    // jobs of an op per half of the tile: (rows x slots) of a job against the half's 2^(m - 1)
    auto jobs_of = [&](int m) { return m - 1 > 7 + SB ? 1 << (m - 1 - 7 - SB) : 1; };
    uint32_t jobs = 0;  // jobs so far: job j uses operand buffer j & 1

    if (warp >= kSpecial / 32) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(SV_TC_WORKER_REGS));
        const int wt = tid - kSpecial, ww = wt >> 5;  // worker thread and warp
        const bool splits = ww < kWorkers / 64;  // else re-assembles
        const int hs = (ww >> 2) & 1, row = (ww & 3) * 32 + (tid & 31);
        const uint32_t tm = tmem + ((uint32_t)((ww & 3) * 32) << 16);
        volatile int* const s_stop = &s_dead;
        bool dead = false;  // a wait has given up: barriers and elementwise ops go on, waits and MMAs do not
        uint32_t dense = 0;      // dense ops so far
        bool preloaded = false;  // the tile's loads were issued while the one before was stored
        // of the entry: this thread's first vector (global address, byte offset in the tile) and its run of 2^c
        // amplitudes; the tiles' positions, in bytes, and their deposit of one step of the grid
        unsigned char* my_g = nullptr;
        int my_s = 0;
        uint64_t my_run = 0, base = 0, others = 0, stride = 0;
        for (uint64_t t = blockIdx.x; t < total_tiles; t += gridDim.x) {
            const bool fresh = enter(t);
            load_chunk(0, chunk_size(0));
            const int m = P.m, n_ops = P.n_ops;
            constexpr uint64_t kAmp = sizeof(Store);
            if (fresh) {
                auto spread = [&](uint64_t v) {  // the bits of v at the positions outside the tile
                    uint64_t d = 0;
                    for (int b = 0; b < P.n - m; b++) d |= ((v >> b) & 1) << P.NL[b];
                    return d * kAmp;
                };
                my_g = reinterpret_cast<unsigned char*>(s_state) + deposit((wt << VS) & ((1 << m) - 1)) * kAmp;
                my_s = swz<SwzT>(wt << VS) * (int)sizeof(Smem);
                my_run = deposit((wt << P.c) & ((1 << m) - 1)) * kAmp;
                others = spread(~0ull);
                stride = spread(gridDim.x);
                base = spread(t - s_begin);
            }
            // adding within the bits of `others`: the carries run through the bits between them
            const uint64_t next = ((base | ~others) + stride) & others;
            const bool more = t + gridDim.x - s_begin < P.tile_count;  // the CTA's next tile belongs to this entry
            const int vecs = 1 << (m - VS), steps = vecs > kWorkers ? vecs / kWorkers : 1;
            const bool mine = wt < vecs;
            const uint32_t sbase = smem_addr(smb);
            auto at_step = [&](int4 q) { return ((uint64_t)(uint32_t)q.y << 32) | (uint32_t)q.x; };
            if (!preloaded && mine) {
                bool raw = true;
                if constexpr (!C64) raw = (P.io & IO_LOAD_Q56) != 0;
                if (raw) {
                    for (int it = 0; it < steps; it++) {
                        const int4 q = s_step[it];
                        cp_async16(sbase + (uint32_t)(my_s ^ q.z), my_g + (base + at_step(q)));
                    }
                } else if constexpr (!C64) {
                    constexpr int U = 4;  // loads in flight per thread before the conversions
                    for (int it = 0; it < steps; it += U) {
                        Cx<double> a[U];
#pragma unroll
                        for (int u = 0; u < U; u++)
                            if (it + u < steps)
                                a[u] = *reinterpret_cast<const Cx<double>*>(my_g + (base + at_step(s_step[it + u])));
#pragma unroll
                        for (int u = 0; u < U; u++)
                            if (it + u < steps)
                                *reinterpret_cast<Smem*>(smb + (my_s ^ s_step[it + u].z)) =
                                    Smem{(unsigned long long)d2q<56>(a[u].re) + t05::kBias,
                                         (unsigned long long)d2q<56>(a[u].im) + t05::kBias};
                    }
                }
            }
            cp_async_wait_all();
            if (more) {
                // the CTA's next tile into L2 while this one is computed: one bulk
                // prefetch per run of 2^c contiguous amplitudes
                const int runs = 1 << (m - P.c);
                for (int r = wt; r < runs; r += kWorkers) {
                    const unsigned char* src = reinterpret_cast<const unsigned char*>(s_state) + next +
                                               (r == wt ? my_run : deposit(r << P.c) * kAmp);
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(src), "r"((int)kAmp << P.c)
                                 : "memory");
                }
            }
            workers_sync();
            bool settle = false;  // an elementwise op's writes are not yet ordered before the next dense op
            auto await = [&](uint32_t mbar, uint32_t parity) {
                if (!dead && !wait(mbar, parity, s_stop)) {
                    give_up(s_stop);
                    dead = true;
                }
            };
            for (int first = 0; first < n_ops; first += kOps) {
                const int nc = chunk_size(first);
                if (n_ops > kOps) load_chunk(first, nc);
                for (int o = 0; o < nc; o++) {
                    const DevOp& op = s_ops[o];
                    if (op.kind == OP_DENSE) {
                        if (settle) workers_sync();
                        settle = false;
                        const uint16_t* tab = s_tab + o * kTabInts;
                        const int kt = kt_of(op), nj = jobs_of(m);
                        constexpr int B = sizeof(Smem);
                        Slots j;
                        const int at = (tab[kTabLane + (tid & 31)] ^ tab[kTabWarp + (ww & 3)]) * B;
                        const int ox = tab[kTabX] * B, orr = tab[kTabR] * B;
                        const int os = tab[kTabWarp + 4] * B, oh = tab[kTabWarp + 8] * B;
#pragma unroll
                        for (int b = 0; b < 3; b++) j.o[b] = tab[kTabSlot + b] * B;
                        // rows that exist in half h, slot bit s (all but in small tiles)
                        auto live = [&](int h, int s) {
                            const int r0 = C64 ? t32::first_row(kt, h, s) : t05::first_row(kt, h, s);
                            return row + r0 < (1 << (m - 1 - kt));
                        };
                        // the thread's slots: splitting, slot bit hs of both halves; re-assembling, half hs
                        const int own = at ^ (hs ? (splits ? os : oh) : 0);
                        if (splits) {
                            const int plane = C64 ? t32::a_plane(kt) : t05::a_plane(kt);
                            for (int x = 0; x < 2; x++) {
                                // what this half's jobs read has been stored (both halves' when p has changed)
                                if (dense > 0) {
                                    await(stored(x), (dense - 1) & 1);
                                    if (x == 0 && s_change[o]) await(stored(1), (dense - 1) & 1);
                                }
                                for (int r = 0; r < nj; r++, jobs++) {
                                    const uint32_t buf = jobs & 1, use = jobs >> 1;
                                    if (use > 0) await(afree(buf), (use - 1) & 1);
                                    if (dead) continue;
                                    fence_after();
                                    const uint32_t a = tm + kACol + kABuf * buf;
#pragma unroll
                                    for (int h = 0; h < 2; h++) {
                                        j.at = own ^ (x ? ox : 0) ^ (r ? orr : 0) ^ (h ? oh : 0);
                                        if constexpr (!C64)
                                            t05::split(smb, j, live(h, hs), a + t05::a_col(kt, h, hs),
                                                       a + t05::a_top(kt, h, hs), plane);
                                        else t32::split(smb, j, live(h, hs), a + t32::a_col(kt, h, hs), plane);
                                    }
                                    st_wait();
                                    warp_arrive(ready(buf));
                                }
                            }
                        } else {
                            const int level = C64 ? t32::acc_level(kt) : t05::acc_level(kt);
                            for (int x = 0; x < 2; x++) {
                                for (int r = 0; r < nj; r++, jobs++) {
                                    await(done(hs), jobs & 1);
                                    if (dead) continue;
                                    fence_after();
#pragma unroll
                                    for (int s = 0; s < 2; s++) {
                                        typename Tr::Words z;
                                        const uint32_t acc = tm + kAccHalf * hs;
                                        if constexpr (!C64) t05::read(acc + t05::acc_col(kt, s), level, z);
                                        else t32::read(acc + t32::acc_col(kt, s), level, z);
                                        ld_wait();
                                        if (s == 1) warp_arrive(accfree(hs, jobs & 1));
                                        j.at = own ^ (x ? ox : 0) ^ (r ? orr : 0) ^ (s ? os : 0);
                                        if (live(hs, s)) {
                                            if constexpr (!C64) t05::store(smb, j, z);
                                            else t32::store(smb, j, z);
                                        }
                                    }
                                }
                                warp_arrive(stored(x));
                            }
                        }
                        dense++;
                    } else {
                        workers_sync();
                        settle = true;
                        const uint4* opc = coef + op.coeff;
                        if (op.kind == OP_PERM) {
                            op_perm<Smem, SwzT>(sm, m, op, opc, s_mv, s_src, wt);
                        } else {
                            // the op's 2^k entries (at most 32) staged in shared memory
                            const unsigned* src = reinterpret_cast<const unsigned*>(opc);
                            unsigned* dst = reinterpret_cast<unsigned*>(s_diag);
                            for (int i = wt; i < (int)(sizeof(typename Tr::DiagEntry) / 4) << op.k; i += kWorkers)
                                dst[i] = src[i];
                            workers_sync();
                            op_diag(sm, m, op, reinterpret_cast<const typename Tr::DiagEntry*>(s_diag), base / kAmp, wt);
                        }
                    }
                }
            }
            workers_sync();
            dead = dead || *s_stop;  // (what is stored then is undefined; the host reports SV_ERR_TIMEOUT)
            // each thread refills its slots with the CTA's next tile by cp.async as soon as it has
            // stored them (same entry, no conversion on load)
            bool raw_in = true, raw_out = true;
            if constexpr (!C64) {
                raw_in = (P.io & IO_LOAD_Q56) != 0;
                raw_out = (P.io & IO_STORE_Q56) != 0;
            }
            const bool refill = more && raw_in;
            if (mine && raw_out) {
                constexpr int U = 4;
                for (int it = 0; it < steps; it += U) {
                    int4 q[U], a[U];
#pragma unroll
                    for (int u = 0; u < U; u++) q[u] = s_step[it + u < steps ? it + u : it];
#pragma unroll
                    for (int u = 0; u < U; u++) a[u] = *reinterpret_cast<const int4*>(smb + (my_s ^ q[u].z));
#pragma unroll
                    for (int u = 0; u < U; u++)
                        if (it + u < steps) *reinterpret_cast<int4*>(my_g + (base + at_step(q[u]))) = a[u];
                    if (!refill) continue;
#pragma unroll
                    for (int u = 0; u < U; u++)
                        if (it + u < steps) cp_async16(sbase + (uint32_t)(my_s ^ q[u].z), my_g + (next + at_step(q[u])));
                }
            } else if constexpr (!C64) {
                for (int it = 0; mine && it < steps; it++) {
                    const int4 q = s_step[it];
                    const Smem b = *reinterpret_cast<const Smem*>(smb + (my_s ^ q.z));
                    *reinterpret_cast<Cx<double>*>(my_g + (base + at_step(q))) =
                        Cx<double>{q2d<56>((long long)(b.re - t05::kBias)), q2d<56>((long long)(b.im - t05::kBias))};
                    if (refill) cp_async16(sbase + (uint32_t)(my_s ^ q.z), my_g + (next + at_step(q)));
                }
            }
            base = next;
            preloaded = refill;
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(SV_TC_ISSUER_REGS));
        volatile int* dead = &s_dead;
        const int role = warp;  // 0, 1: issue the MMAs of even, odd jobs; 2: copies the block images
        const uint32_t b0 = smem_addr(smraw);
        unsigned d = 0;  // dense ops so far; op d's image is in buffer d & 1
        auto await = [&](uint32_t mbar, uint32_t parity) {
            if (wait(mbar, parity, dead)) return true;
            give_up(dead);
            return false;
        };
        for (uint64_t t = blockIdx.x; t < total_tiles; t += gridDim.x) {
            enter(t);
            load_chunk(0, chunk_size(0));
            const int n_ops = P.n_ops, m = P.m;
            for (int first = 0; first < n_ops; first += kOps) {
                const int nc = chunk_size(first);
                if (n_ops > kOps) load_chunk(first, nc);
                for (int o = 0; o < nc; o++) {
                    if (s_ops[o].kind != OP_DENSE || role > 2 || *dead) continue;
                    const int kt = kt_of(s_ops[o]);
                    const int buf = d & 1;
                    const uint32_t use = d >> 1;  // earlier uses of this buffer
                    d++;
                    if (role == 2) {
                        if (use > 0 && !await(bfree(buf), (use - 1) & 1)) continue;
                        const int bytes = C64 ? t32::image_bytes(kt) : t05::image_bytes(kt);
                        if (elect_one())
                            bulk_load(b0 + buf * Tr::kBBytes, image_at(coef, s_ops[o].coeff), (uint32_t)bytes, bfull(buf));
                        __syncwarp();
                        continue;
                    }
                    if (!await(bfull(buf), use & 1)) continue;
                    const int nj = 2 * jobs_of(m);  // even
                    const bool stall = (s_ops[o].flags & OPF_TEST_NO_MMA) != 0;
                    // (blocks narrower than the slots fill the second half with further groups, if there are any)
                    const bool two = kt == SB || m - 1 > 7 + SB - 1;
                    const uint32_t b = b0 + buf * Tr::kBBytes;
                    auto issue_half = [&](auto H) {
                        if constexpr (C64) {
                            if (role == 0) t32::issue_any<H.value, 0>(kt, b);
                            else t32::issue_any<H.value, 1>(kt, b);
                        } else {
                            if (role == 0) t05::issue_any<H.value, 0>(kt, b);
                            else t05::issue_any<H.value, 1>(kt, b);
                        }
                    };
                    for (int r = role; r < nj; r += 2) {
                        const uint32_t j = jobs + r;  // operand buffer j & 1 = role
                        if (!await(ready(role), (j >> 1) & 1)) break;
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            // job j - 1's re-assembly has read the accumulator
                            if (j > 0 && !await(accfree(h, role ^ 1), ((j - 1) >> 1) & 1)) break;
                            fence_after();
                            if (elect_one()) {
                                // (OPF_TEST_NO_MMA, a test hook: nothing is issued, so the workers' bounded wait runs out)
                                if (!stall) {
                                    if (h == 0) issue_half(Int<0>{});
                                    else if (two) issue_half(Int<1>{});
                                    commit(done(h));
                                }
                                if (h == 1) {
                                    commit(afree(role));
                                    if (r + 2 >= nj) commit(bfree(buf));
                                }
                            }
                            __syncwarp();
                        }
                    }
                    jobs += nj;
                }
            }
        }
        // nothing of this CTA's may be in flight when it leaves: the last image, the MMAs
        if (role == 2) {
            for (unsigned i = d > 2 ? d - 2 : 0; i < d; i++) wait(bfull(i & 1), (i >> 1) & 1, dead);
        } else if (role < 2) {
            if (elect_one()) commit(end_bar);
            __syncwarp();
            int never = 0;
            wait(end_bar, 0, &never);
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// ---------------------------------------------------------------------------
// Launcher.
// ---------------------------------------------------------------------------
template <bool C64>
static cudaError_t launch_tc(const BatchEntry* d_entries, int n_entries, uint64_t total_tiles, int max_m,
                             const DevOp* d_ops, const void* d_coef, cudaStream_t s, const DevInfo& di) {
    using Tr = TcMode<C64>;
    const size_t smem =
        std::max<size_t>(2 * Tr::kBBytes + ((size_t)1 << max_m) * sizeof(typename Tr::Smem), tc::kSmemMin);
    static std::atomic<size_t> dyn_max[64];  // per device: opt-in limit minus the kernel's static shared memory
    size_t most = dyn_max[di.device].load();
    if (most == 0) {
        cudaFuncAttributes fa{};
        cudaError_t e = cudaFuncGetAttributes(&fa, k_tile_pass_tc<C64>);
        if (e != cudaSuccess) return e;
        most = di.smem_optin - fa.sharedSizeBytes;
        e = cudaFuncSetAttribute(k_tile_pass_tc<C64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
        if (e != cudaSuccess) return e;
        dyn_max[di.device].store(most);
    }
    if (smem > most) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)std::min<uint64_t>((uint64_t)di.sms, total_tiles);
    k_tile_pass_tc<C64><<<grid, tc::kCta, smem, s>>>(d_entries, n_entries, total_tiles, d_ops, (const uint4*)d_coef);
    return cudaGetLastError();
}

// Block images, one CTA each.
template <bool C64>
__global__ void k_block_images(const ImageJob* __restrict__ jobs, uint4* __restrict__ coef) {
    const ImageJob j = jobs[blockIdx.x];
    const double2* M = reinterpret_cast<const double2*>(coef + j.matrix);
    unsigned char* img = const_cast<unsigned char*>(tc::image_at(coef, j.image));
    if constexpr (C64) t32::build_image(M, img, j.k);
    else t05::build_image(M, img, j.k);
}

static_assert(t05::image_bytes(3) % kImageUnit == 0 && t05::image_bytes(4) % kImageUnit == 0 &&
                  t32::image_bytes(3) % kImageUnit == 0 && t32::image_bytes(4) % kImageUnit == 0 &&
                  t32::image_bytes(5) % kImageUnit == 0,
              "images lie one behind another in whole units");
size_t block_image_bytes(int dt, int k) { return dt == SV_C64 ? t32::image_bytes(k) : t05::image_bytes(k); }

cudaError_t launch_block_images(int dt, const ImageJob* d_jobs, int n, void* d_coef, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (dt == SV_C64) k_block_images<true><<<n, 256, 0, s>>>(d_jobs, (uint4*)d_coef);
    else k_block_images<false><<<n, 256, 0, s>>>(d_jobs, (uint4*)d_coef);
    return cudaGetLastError();
}

cudaError_t launch_tile_pass_tc(int dt, const BatchEntry* d_entries, int n_entries, uint64_t total_tiles, int max_m,
                                const DevOp* d_ops, const void* d_coef, cudaStream_t s, const DevInfo& di) {
    return dt == SV_C64 ? launch_tc<true>(d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di)
                        : launch_tc<false>(d_entries, n_entries, total_tiles, max_m, d_ops, d_coef, s, di);
}

cudaError_t tc_fault_take(int* fault) {
    int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(fault, tc::g_fault, sizeof(int));
    if (e == cudaSuccess && *fault) e = cudaMemcpyToSymbol(tc::g_fault, &zero, sizeof(int));
    return e;
}

}  // namespace svk
