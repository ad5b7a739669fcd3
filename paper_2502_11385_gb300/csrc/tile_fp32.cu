// K5-fp32: the tile pass on the FP32 pipe, complex64 in float32 and complex128
// in double-float pairs (the arithmetic is in tile_common.cuh).
//
// These modes run the small states (by default below 23 and 20 qubits), where a
// pass has no more tiles than there are SMs and a tile's ops follow one another
// through barriers, so an op's latency counts as much as its
// work.  The tile is held twice in shared memory and every dense and permutation
// op goes from one copy to the other, one thread per output amplitude (two or
// four rows in float32, where each amplitude loaded then serves them all): an
// output needs its group's 2^k amplitudes and one row of the block, nothing is
// kept in registers across a barrier, an op has one barrier, and 64 registers let
// 1024 threads share the tile.  The coefficients of the next op arrive in shared
// memory while the current one runs.  What bounds it: the FP32 and integer issue
// slots of the SMs that have a tile.
//
// While a pass has fewer tiles than SMs, a cluster of 2, 4 or 8 CTAs shares each
// tile: its highest positions number the CTA, an output is formed in the CTA that
// holds it, and a block on those positions reads its other amplitudes from their
// CTAs' shared memory.  The plan, its passes and the sums stay as they are.  A
// barrier of the cluster divides two ops if either reads another CTA, else the
// CTA's own does.  Clusters are taken no larger than all of a launch's run at once
// (16 clusters of 8 do not: 16 qubits complex128 253 us, as 16 of 4 it is one wave).
//
// Against k_tile_pass's one thread per group of 2^k amplitudes (256 threads of
// 140 registers and more), kernel time of a circuit: complex128 brickwork of 10
// layers, 10 qubits 125 -> 58 us, 12: 283 -> 86, 15: 380 -> 128, 17: 440 -> 193,
// 19 (128 tiles, no clusters): 508 -> 451; complex64 11 qubits 66 -> 47,
// 13: 138 -> 70, 16: 186 -> 104, 18: 213 -> 150.  Once SMs have several tiles
// k_tile_pass is the better one again: three of its CTAs overlap one's loads and
// stores with another's ops (25 qubits complex64: a pass without ops 3.8 ps an
// amplitude against 4.8, a one-qubit block 0.9 against 1.4, though a 3-qubit block
// 3.2 against 2.3; a 21-qubit QAOA of 256 tiles 270 us against 347).  So this
// kernel takes launches of up to one tile an SM, and of up to four where the
// pass's ops cost less here by those figures (complex64, `few`: passes of 3-qubit
// blocks, 21 qubits 571 -> 441 us a circuit, 22 qubits 1120 -> 889).  Among the many
// states of a batch wide blocks cost k_tile_pass more than they do there, so a batch's
// launch of any number of tiles of 2^10 amplitudes and more takes the kernel that its
// ops cost less with (`few`; by the batch costs in api.cu: 304 states of 14 qubits,
// 3-qubit blocks 1.23 times as fast here, 4-qubit ones 1.37, one-qubit gates 0.81 times;
// complex128 1.16, 1.19, 0.89).  Both give the same bits (each sum in the same order).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "kernels.cuh"
#include "sv.h"
#include "tile_common.cuh"

namespace svk {

namespace fp32 {

constexpr int kOps = 48;         // op descriptors held per pass
constexpr int kCoefs = 1056;     // staged coefficients of an op: 2^5 rows and their padding
constexpr int kMaxThreads = 1024;
constexpr int kSteps = 4;       // log2 of the outputs a thread forms in one op at most (one row each)
constexpr int kMaxCluster = 3;  // log2 of the CTAs that share a tile
constexpr int kMinSlice = 8;    // log2 of the amplitudes a CTA of a cluster holds at least
// The smallest tile that a cluster shares: below it a CTA's share of an op is less than the
// cluster's barrier (complex64, 2^10 amplitudes: 37 us alone, 41 as four CTAs; 2^11: 58 and 47).
template <bool DF>
constexpr int kClusterTile = DF ? 9 : 11;
template <bool DF>
constexpr int kMaxTile = DF ? 12 : 13;  // two copies of a tile and the staged coefficients: 165 or 148 KB

template <bool DF>
struct Mode;
template <>
struct Mode<false> {
    using Store = Cx<float>;
    using Smem = Cx<float>;
    using SwzT = float;
};
template <>
struct Mode<true> {
    using Store = Cx<double>;
    using Smem = DF4;
    using SwzT = double;
};

__device__ __forceinline__ Cx<float> turn(Cx<float> v, int c) { return rot_i(v, c); }
__device__ __forceinline__ DF4 turn(DF4 v, int c) { return rot_df(v, c); }
__device__ __forceinline__ int move_of(const Cx<float>* M, int t) { return (int)M[t].re; }
__device__ __forceinline__ int move_of(const DF4* M, int t) { return (int)M[t].rh; }

// One row of a block product: acc starts with column 0 and takes the columns in order.
struct Sum32 {
    float re, im;
    __device__ __forceinline__ void first(Cx<float> u, Cx<float> a) {
        re = im = 0.f;
        next(u, a);
    }
    __device__ __forceinline__ void next(Cx<float> u, Cx<float> a) {
        re = fmaf(u.re, a.re, re);
        re = fmaf(-u.im, a.im, re);
        im = fmaf(u.re, a.im, im);
        im = fmaf(u.im, a.re, im);
    }
    __device__ __forceinline__ Cx<float> value() const { return Cx<float>{re, im}; }
};
struct SumDf {
    float rh, rl, ih, il;
    __device__ __forceinline__ void first(DF4 u, DF4 a) {
        df_mul(rh, rl, u.rh, u.rl, a.rh, a.rl);
        df_mac(rh, rl, -u.ih, -u.il, a.ih, a.il);
        df_mul(ih, il, u.rh, u.rl, a.ih, a.il);
        df_mac(ih, il, u.ih, u.il, a.rh, a.rl);
    }
    __device__ __forceinline__ void next(DF4 u, DF4 a) {
        df_mac(rh, rl, u.rh, u.rl, a.rh, a.rl);
        df_mac(rh, rl, -u.ih, -u.il, a.ih, a.il);
        df_mac(ih, il, u.rh, u.rl, a.ih, a.il);
        df_mac(ih, il, u.ih, u.il, a.rh, a.rl);
    }
    __device__ __forceinline__ DF4 value() {
        df_norm(rh, rl);
        df_norm(ih, il);
        return DF4{rh, rl, ih, il};
    }
};
__device__ __forceinline__ Cx<float> phase(Cx<float> u, Cx<float> a) {
    return Cx<float>{fmaf(u.re, a.re, -u.im * a.im), fmaf(u.re, a.im, u.im * a.re)};
}
__device__ __forceinline__ DF4 phase(DF4 u, DF4 a) {
    SumDf s;
    s.first(u, a);
    return s.value();
}
__device__ __forceinline__ Cx<float> negate(Cx<float> a) { return Cx<float>{-a.re, -a.im}; }
__device__ __forceinline__ DF4 negate(DF4 a) { return DF4{-a.rh, -a.rl, -a.ih, -a.il}; }
__device__ __forceinline__ bool negative(Cx<float> u) { return u.re < 0.f; }
__device__ __forceinline__ bool negative(DF4 u) { return u.rh < 0.f; }

// Addresses of an op, formed once per pass: swz() is linear over XOR, so the
// shared-memory index of (amplitude ^ bits) is the index ^ swz(bits).
//
// A thread forms the outputs it | at of a thread part `it` and a part `at` in the
// tile's highest positions that is the same for all threads and counts in Gray
// code: a step changes one position, three XORs with the step's entry.  (Integer
// instructions run at half the FP32 rate; with the indices formed anew for each
// output they were the bound: 25 qubits complex64, a diagonal 2.2 ps an amplitude
// against 1.2, a permutation 2.9 against 1.6.)
struct Step {
    int base, to;  // swz of the position: outside the block only, and any
    int row, pad;  // its bit of the block's row
};
struct alignas(16) OpAt {
    int sp[5];      // swz of the block's tile positions (0 where the op has none)
    int block;      // the block's positions
    int skip;       // those of the rows one thread forms (dense)
    int count, tb;  // values of the common part; positions of the thread part
    int far;        // the block's positions that number a CTA of the cluster, as its rank's bits
    int pad[2];
    Step step[kSteps];
};

template <typename SwzT>
__device__ OpAt op_at(const DevOp& op, int m, int rows, int threads) {
    OpAt a{};
    for (int j = 0; j < 5; j++)
        if (j < op.k && op.pos[j] >= m) {
            if (op.kind != OP_DIAG) a.far |= 1 << (op.pos[j] - m);
        } else if (j < op.k && op.pos[j] >= 0) {
            a.sp[j] = swz<SwzT>(1 << op.pos[j]);
            a.block |= 1 << op.pos[j];
            if (op.kind == OP_DENSE && (1 << j) < rows) a.skip |= 1 << op.pos[j];
        }
    const int bits = m - __popc(a.skip);
    a.tb = min(bits, 31 - __clz(threads));
    int h = bits - a.tb;  // at most kSteps: the launch has 2^(m - kSteps) threads or more
    a.count = 1 << h;
    for (int b = m - 1; h > 0; b--)
        if (!((a.skip >> b) & 1)) {
            Step& s = a.step[--h];
            s.to = swz<SwzT>(1 << b);
            s.base = (a.block >> b) & 1 ? 0 : s.to;
            for (int j = 0; j < 5; j++)
                if (j < op.k && op.pos[j] == b) s.row = 1 << j;
        }
    return a;
}

// The thread part of a thread's outputs: its number with zeros put in at `skip`.
__device__ __forceinline__ int thread_part(const OpAt& a) {
    int it = threadIdx.x & ((1 << a.tb) - 1);
    for (int left = a.skip; left; left &= left - 1) it += it & -(left & -left);
    return it;
}

// f(base, to, row) for each value of the common part, from the thread part's values.
template <typename F>
__device__ __forceinline__ void each(const OpAt& a, int base, int to, int row, F f) {
    if ((int)threadIdx.x >> a.tb) return;
    const int count = a.count;
#pragma unroll 1
    for (int q = 1;; q++) {
        f(base, to, row);
        if (q == count) break;
        const Step s = a.step[__ffs(q) - 1];
        base ^= s.base;
        to ^= s.to;
        row ^= s.row;
    }
}

template <int K>
__device__ __forceinline__ int row_of(int i, const DevOp& op) {
    int row = 0;
#pragma unroll
    for (int j = 0; j < K; j++) row |= ((i >> op.pos[j]) & 1) << j;
    return row;
}

// Where U[row][col] of a block of 2^k rows lies among the staged coefficients:
// the RT rows of a thread side by side, 16 bytes of padding after each RT rows
// (threads of a warp may hold different rows).
template <int RT>
__device__ __forceinline__ int staged_at(int row, int col, int k) {
    constexpr int pad = RT == 1 ? 1 : 2;
    return (row / RT) * ((RT << k) + pad) + col * RT + row % RT;
}

// out = U in on every group of 2^K amplitudes; M: U as staged_at<RT> lays it.  A
// thread forms RT rows that differ in the block's lowest positions.
template <int K, bool DF, int RT>
__device__ __forceinline__ void dense(const typename Mode<DF>::Smem* in, typename Mode<DF>::Smem* out,
                                      const DevOp& op, const OpAt& oa, const typename Mode<DF>::Smem* M) {
    using T = Mode<DF>;
    using S = typename T::Smem;
    using SwzT = typename T::SwzT;
    constexpr int D = 1 << K;
    struct alignas(16) Rows {
        S v[RT];
    };
    int sp[K];
#pragma unroll
    for (int j = 0; j < K; j++) sp[j] = oa.sp[j];
    auto off = [&](int c) {
        int o = 0;
#pragma unroll
        for (int j = 0; j < K; j++)
            if ((c >> j) & 1) o ^= sp[j];
        return o;
    };
    const int it = thread_part(oa);
    each(oa, swz<SwzT>(it & ~oa.block), swz<SwzT>(it), row_of<K>(it, op),
         [&](int base, int to, int row) {
            const S* u = M + staged_at<RT>(row, 0, K);
            typename std::conditional<DF, SumDf, Sum32>::type s[RT];
#pragma unroll(K <= 3 ? D : 8)
            for (int c = 0; c < D; c++) {
                const S a = in[base ^ off(c)];
                Rows w;
                if constexpr (RT == 1) w.v[0] = u[c];
                else w = *reinterpret_cast<const Rows*>(u + c * RT);
#pragma unroll
                for (int r = 0; r < RT; r++) {
                    if (c == 0) s[r].first(w.v[r], a);
                    else s[r].next(w.v[r], a);
                }
            }
#pragma unroll
            for (int r = 0; r < RT; r++) out[to ^ off(r)] = s[r].value();
         });
}

// The element `at` of the CTA of rank `rank` in this cluster's copies of `local`.
template <typename S>
__device__ __forceinline__ S load_far(const S* local, int at, int rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(local + at)), "r"(rank));
    S v;
    if constexpr (sizeof(S) == 16)
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.rh), "=f"(v.rl), "=f"(v.ih), "=f"(v.il)
                     : "r"(a));
    else
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.re), "=f"(v.im) : "r"(a));
    return v;
}

// Bits of the block's row that this CTA's rank fixes; lm: positions of a slice.
__device__ __forceinline__ int far_row(const DevOp& op, int lm, int rank) {
    int row = 0;
#pragma unroll
    for (int j = 0; j < 5; j++)
        if (j < op.k && op.pos[j] >= lm) row |= ((rank >> (op.pos[j] - lm)) & 1) << j;
    return row;
}

// dense() for a block with positions beyond the slice: a column's amplitude comes
// from the CTA that holds it, outputs stay here.
template <int K, bool DF>
__device__ __forceinline__ void dense_far(const typename Mode<DF>::Smem* in, typename Mode<DF>::Smem* out,
                                          const DevOp& op, const OpAt& oa, const typename Mode<DF>::Smem* M, int lm,
                                          int rank) {
    using SwzT = typename Mode<DF>::SwzT;
    using S = typename Mode<DF>::Smem;
    constexpr int D = 1 << K;
    int sp[K], fp[K];  // a block position within the slice, or among the ranks
#pragma unroll
    for (int j = 0; j < K; j++) {
        sp[j] = oa.sp[j];
        fp[j] = op.pos[j] >= lm ? 1 << (op.pos[j] - lm) : 0;
    }
    const int it = thread_part(oa);
    each(oa, swz<SwzT>(it & ~oa.block), swz<SwzT>(it), row_of<K>(it, op) | far_row(op, lm, rank),
         [&](int base, int to, int row) {
             const S* u = M + staged_at<1>(row, 0, K);
             typename std::conditional<DF, SumDf, Sum32>::type s;
#pragma unroll(K <= 3 ? D : 8)
             for (int c = 0; c < D; c++) {
                 int at = base, rk = rank & ~oa.far;
#pragma unroll
                 for (int j = 0; j < K; j++)
                     if ((c >> j) & 1) {
                         at ^= sp[j];
                         rk |= fp[j];
                     }
                 const S a = load_far(in, at, rk);
                 if (c == 0) s.first(u[0], a);
                 else s.next(u[c], a);
             }
             out[to] = s.value();
         });
}

// out[r] = i^code(r) in[src(r)] inside every group; table[r] = the shared-memory
// offset of src(r) in its group | code << 16 | the rank's bits of src(r) << 20.
template <bool DF, bool CL>
__device__ __forceinline__ void permute(const typename Mode<DF>::Smem* in, typename Mode<DF>::Smem* out, const DevOp& op,
                                        const OpAt& oa, const int* table, int lm, int rank) {
    using SwzT = typename Mode<DF>::SwzT;
    const int it = threadIdx.x;
    int row = CL ? far_row(op, lm, rank) : 0;
#pragma unroll
    for (int j = 0; j < 5; j++)
        if (j < op.k) row |= ((it >> op.pos[j]) & 1) << j;
    each(oa, swz<SwzT>(it & ~oa.block), swz<SwzT>(it), row, [&](int base, int to, int row) {
        const int e = table[row], at = base ^ (e & 0xffff);
        if (CL && oa.far) out[to] = turn(load_far(in, at, (rank & ~oa.far) | e >> 20), (e >> 16) & 3);
        else out[to] = turn(in[at], (e >> 16) & 3);
    });
}

// a <- u a in place, u chosen by the op's bits of the amplitude's index.
template <bool DF>
__device__ __forceinline__ void diagonal(typename Mode<DF>::Smem* sm, const DevOp& op, const OpAt& oa,
                                         const typename Mode<DF>::Smem* M, uint64_t tile_base, int lm, int rank) {
    using SwzT = typename Mode<DF>::SwzT;
    const int it = threadIdx.x;
    int row = 0;
#pragma unroll
    for (int j = 0; j < 5; j++)
        if (j < op.k)
            row |= (op.pos[j] < 0     ? (int)((tile_base >> op.qbit[j]) & 1)
                    : op.pos[j] >= lm ? (rank >> (op.pos[j] - lm)) & 1
                                      : (it >> op.pos[j]) & 1)
                   << j;
    if (op.flags & OPF_SIGN_ONLY)
        each(oa, 0, swz<SwzT>(it), row, [&](int, int to, int row) {
            if (negative(M[row])) sm[to] = negate(sm[to]);
        });
    else
        each(oa, 0, swz<SwzT>(it), row, [&](int, int to, int row) { sm[to] = phase(M[row], sm[to]); });
}

template <typename S>
__device__ __forceinline__ void copy_async(S* dst, const S* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(sizeof(S))
                 : "memory");
}

__device__ __forceinline__ void sync_cluster() {
    asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
}

}  // namespace fp32

// CL: a cluster of 2^lc CTAs shares a tile (RT = 1); each holds the slice whose
// highest lc positions are its rank.
template <bool DF, int RT, bool CL>
__global__ void __launch_bounds__(CL ? fp32::kMaxThreads / 2 : fp32::kMaxThreads, 1)
    k_tile_pass_fp32(const BatchEntry* __restrict__ E, int n_entries, uint64_t total_tiles,
                     const DevOp* __restrict__ ops, const typename fp32::Mode<DF>::Smem* __restrict__ coef,
                     int lc) {
    using namespace fp32;
    using T = Mode<DF>;
    using S = typename T::Smem;
    using Store = typename T::Store;
    using SwzT = typename T::SwzT;
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ uint64_t dep[2][32];  // deposit tables for the tile's high local bits
    __shared__ __align__(16) DevPass P;
    __shared__ uint64_t s_state, s_begin;
    __shared__ DevOp s_ops[kOps];
    __shared__ OpAt s_at[kOps];
    __shared__ __align__(16) S s_coef[2][kCoefs];  // the current and the next op's coefficients
    __shared__ int s_perm[2][32];                  // or permutation table
    const int tid = threadIdx.x, nt = blockDim.x;
    const int rank = CL ? blockIdx.x & ((1 << lc) - 1) : 0;
    if constexpr (!CL) lc = 0;
    // descriptors of ops [o, o + count) of the pass and their addresses
    auto load_ops = [&](int o, int count) {
        const int4* src = reinterpret_cast<const int4*>(ops + P.op0 + o);
        int4* dst = reinterpret_cast<int4*>(s_ops);
        for (int i = tid; i < count * (int)(sizeof(DevOp) / 16); i += nt) dst[i] = src[i];
        for (int i = tid; i < count; i += nt) {
            const DevOp& op = ops[P.op0 + o + i];
            s_at[i] = op_at<SwzT>(op, P.m - lc, op.k == 1 && RT > 2 ? 2 : RT, nt);
        }
    };
    int cur = -1;
    for (uint64_t t = blockIdx.x >> lc; t < total_tiles; t += gridDim.x >> lc) {
        if (cur < 0 || t - s_begin >= P.tile_count) {
            int lo = cur < 0 ? 0 : cur, hi = n_entries - 1;  // entry owning tile t (uniform across the CTA)
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (E[mid].tile_begin <= t) lo = mid;
                else hi = mid - 1;
            }
            __syncthreads();
            const unsigned* src = reinterpret_cast<const unsigned*>(&E[lo].p);
            unsigned* dst = reinterpret_cast<unsigned*>(&P);
            for (int i = tid; i < (int)(sizeof(DevPass) / 4); i += nt) dst[i] = src[i];
            if (tid == 0) {
                s_state = E[lo].state;
                s_begin = E[lo].tile_begin;
            }
            __syncthreads();
            if (P.n_ops <= kOps) load_ops(0, P.n_ops);
            if (tid < 64) {
                const int w = tid >> 5, v = tid & 31;
                uint64_t d = 0;
                for (int b = 0; b < 5; b++) {
                    const int j = P.c + 5 * w + b;
                    if (j < P.m && ((v >> b) & 1)) d |= 1ull << P.L[j];
                }
                dep[w][v] = d;
            }
            __syncthreads();
            cur = lo;
        }
        Store* const st = reinterpret_cast<Store*>(s_state);
        const int m = P.m - lc, c = P.c, n_ops = P.n_ops;  // m: positions of this CTA's slice
        const int cmask = (1 << c) - 1;
        S* in = reinterpret_cast<S*>(smraw);
        S* out = in + (1 << m);
        uint64_t base = 0;
        for (int b = 0; b < P.n - P.m; b++) base |= (((t - s_begin) >> b) & 1) << P.NL[b];
        auto place = [&](int j) {  // global index of the slice's index j
            if constexpr (CL) j |= rank << m;
            const int r = j >> c;
            return base | dep[0][r & 31] | dep[1][(r >> 5) & 31] | (uint64_t)(j & cmask);
        };
        // The coefficients of op o go into buffer o & 1: stage() starts the copies,
        // staged() completes them (before the barrier that precedes op o).
        int move = 0;  // a permutation's row in cycle order, held by the first warp's lanes
        auto stage = [&](int o) {
            const DevOp& op = s_ops[o];
            const S* M = coef + op.coeff;
            const int k = op.k, D = 1 << k;
            if (op.kind == OP_PERM) {
                if (tid < D) move = move_of(M, tid);
                return;
            }
            const int count = op.kind == OP_DIAG ? D : D * D;
            for (int i = tid; i < count; i += nt) {
                const int at = op.kind == OP_DIAG ? i
                               : k == 1           ? staged_at<(RT > 2 ? 2 : RT)>(i >> k, i & (D - 1), k)
                                                  : staged_at<RT>(i >> k, i & (D - 1), k);
                copy_async(&s_coef[o & 1][at], M + i);
            }
        };
        auto staged = [&](int o) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            const DevOp& op = s_ops[o];
            if (op.kind != OP_PERM || tid >= 32) return;
            // row a_t takes its amplitude from the next row of its cycle
            const unsigned ends = __ballot_sync(~0u, tid < (1 << op.k) && (move & 128));
            const unsigned before = ends & ((1u << tid) - 1);
            const int next = (move & 128) ? (before ? 32 - __clz(before) : 0) : tid + 1;
            const int src = __shfl_sync(~0u, move, next);
            int off = 0;
            for (int j = 0; j < 5; j++)
                if ((src >> j) & 1) {
                    off ^= s_at[o].sp[j];
                    if (CL && j < op.k && op.pos[j] >= m) off |= 1 << (20 + op.pos[j] - m);
                }
            if (tid < (1 << op.k)) s_perm[o & 1][move & 31] = off | ((move >> 5) & 3) << 16;
        };
        if (n_ops > 0 && n_ops <= kOps) stage(0);
        if constexpr (DF) {
#pragma unroll 4
            for (int j = tid; j < (1 << m); j += nt) {
                const Cx<double> a = st[place(j)];
                DF4 v;
                d2df(a.re, v.rh, v.rl);
                d2df(a.im, v.ih, v.il);
                in[swz<double>(j)] = v;
            }
        } else {
#pragma unroll 4
            for (int j = 2 * tid; j < (1 << m); j += 2 * nt)
                *reinterpret_cast<int4*>(in + swz<float>(j)) = *reinterpret_cast<const int4*>(st + place(j));
        }
        for (int first = 0; first < n_ops; first += kOps) {
            const int count = min(kOps, n_ops - first);
            if (n_ops > kOps) {  // descriptors in turns
                __syncthreads();
                load_ops(first, count);
                __syncthreads();
                stage(0);
            }
            staged(0);
            if (CL) sync_cluster();
            else __syncthreads();
            for (int o = 0; o < count; o++) {
                const DevOp& op = s_ops[o];
                const OpAt& oa = s_at[o];
                const S* M = s_coef[o & 1];
                if (o + 1 < count) stage(o + 1);
                if (op.kind == OP_DIAG) {
                    diagonal<DF>(in, op, oa, M, base, m, rank);
                } else {
                    if (op.kind == OP_PERM) permute<DF, CL>(in, out, op, oa, s_perm[o & 1], m, rank);
                    else if (CL && oa.far) {
                        if (op.k == 1) dense_far<1, DF>(in, out, op, oa, M, m, rank);
                        else if (op.k == 2) dense_far<2, DF>(in, out, op, oa, M, m, rank);
                        else if (op.k == 3) dense_far<3, DF>(in, out, op, oa, M, m, rank);
                        else if (op.k == 4) dense_far<4, DF>(in, out, op, oa, M, m, rank);
                        else dense_far<5, DF>(in, out, op, oa, M, m, rank);
                    } else if (op.k == 1) dense<1, DF, (RT > 2 ? 2 : RT)>(in, out, op, oa, M);
                    else if (op.k == 2) dense<2, DF, RT>(in, out, op, oa, M);
                    else if (op.k == 3) dense<3, DF, RT>(in, out, op, oa, M);
                    else if (op.k == 4) dense<4, DF, RT>(in, out, op, oa, M);
                    else dense<5, DF, RT>(in, out, op, oa, M);
                    S* const x = in;
                    in = out;
                    out = x;
                }
                if (o + 1 < count) staged(o + 1);
                // other CTAs read this slice for op o (its copy is written next) or will for o + 1
                if (CL && (o + 1 == count || oa.far || s_at[o + 1].far)) sync_cluster();
                else __syncthreads();
            }
        }
        if constexpr (DF) {
#pragma unroll 4
            for (int j = tid; j < (1 << m); j += nt) {
                const DF4 v = in[swz<double>(j)];
                st[place(j)] = Cx<double>{df2d(v.rh, v.rl), df2d(v.ih, v.il)};
            }
        } else {
#pragma unroll 4
            for (int j = 2 * tid; j < (1 << m); j += 2 * nt)
                *reinterpret_cast<int4*>(st + place(j)) = *reinterpret_cast<const int4*>(in + swz<float>(j));
        }
        __syncthreads();
    }
}

// Launch configuration for tiles of 2^max_m amplitudes, 2^lc CTAs each.
template <bool DF, int RT, bool CL>
struct Launch {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute cluster{};
    Launch(uint64_t tiles, uint64_t most_tiles, int max_m, int lc, cudaStream_t s) {
        constexpr int most = CL ? fp32::kMaxThreads / 2 : fp32::kMaxThreads;
        cfg.gridDim = dim3((unsigned)(std::min(tiles, most_tiles) << lc));
        static_assert(most << fp32::kSteps >= 1 << fp32::kMaxTile<DF>, "Step entries cover a thread's outputs");
        cfg.blockDim = dim3(std::min(most, std::max(64, (1 << (max_m - lc)) / RT)));
        cfg.dynamicSmemBytes = 2 * ((size_t)1 << (max_m - lc)) * sizeof(typename fp32::Mode<DF>::Smem);
        cfg.stream = s;
        cluster.id = cudaLaunchAttributeClusterDimension;
        cluster.val.clusterDim.x = 1u << lc;
        cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
        cfg.attrs = &cluster;
        cfg.numAttrs = CL ? 1 : 0;
    }
};

template <bool DF, int RT, bool CL>
static cudaError_t prepare(const DevInfo& di) {
    static std::atomic<bool> ready[64];  // per device
    if (ready[di.device].load()) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(k_tile_pass_fp32<DF, RT, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             2 * (int)sizeof(typename fp32::Mode<DF>::Smem) << fp32::kMaxTile<DF>);
    if (e == cudaSuccess) ready[di.device].store(true);
    return e;
}

template <bool DF, int RT, bool CL>
static cudaError_t launch_fp32(const BatchEntry* d_entries, int n_entries, uint64_t total_tiles, int max_m, int lc,
                               const DevOp* d_ops, const void* d_coef, cudaStream_t s, const DevInfo& di) {
    const cudaError_t e = prepare<DF, RT, CL>(di);
    if (e != cudaSuccess) return e;
    Launch<DF, RT, CL> l(total_tiles, (uint64_t)di.sms, max_m, lc, s);
    return cudaLaunchKernelEx(&l.cfg, k_tile_pass_fp32<DF, RT, CL>, d_entries, n_entries, total_tiles, d_ops,
                              (const typename fp32::Mode<DF>::Smem*)d_coef, lc);
}

// Clusters of 2^lc CTAs that run at once, with the most threads and shared memory
// such a CTA may take (0 where the query fails: no clusters then).
template <bool DF>
static int clusters_at_once(int lc, const DevInfo& di) {
    static std::atomic<int> known[64][fp32::kMaxCluster + 1];  // 1 + the answer
    int v = known[di.device][lc].load();
    if (v == 0) {
        int count = 0;
        Launch<DF, 1, true> l(1, 1, fp32::kMaxTile<DF>, lc, nullptr);
        if (prepare<DF, 1, true>(di) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&count, k_tile_pass_fp32<DF, 1, true>, &l.cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            count = 0;
        }
        v = count + 1;
        known[di.device][lc].store(v);
    }
    return v - 1;
}

template <bool DF>
static int cluster_of(uint64_t total_tiles, int max_m, const DevInfo& di) {
    int lc = 0;
    while (lc < fp32::kMaxCluster && max_m >= fp32::kClusterTile<DF> && max_m - (lc + 1) >= fp32::kMinSlice &&
           total_tiles <= (uint64_t)clusters_at_once<DF>(lc + 1, di))
        lc++;
    return lc;
}

bool tile_pass_fp32_fits(int dt, uint64_t total_tiles, int max_m, bool few, const DevInfo& di) {
    return (few || total_tiles <= (uint64_t)di.sms) &&
           max_m <= (dt == SV_C64 ? fp32::kMaxTile<false> : fp32::kMaxTile<true>);
}

cudaError_t launch_tile_pass_fp32(int dt, const BatchEntry* d_entries, int n_entries, uint64_t total_tiles, int max_m,
                                  const DevOp* d_ops, const void* d_coef, cudaStream_t s, const DevInfo& di) {
    // a cluster for each tile while they all run at once (one entry: its tile is max_m)
    const int lc = n_entries != 1 ? 0
                   : dt == SV_C64 ? cluster_of<false>(total_tiles, max_m, di)
                                  : cluster_of<true>(total_tiles, max_m, di);
    if (lc > 0)
        return dt == SV_C64 ? launch_fp32<false, 1, true>(d_entries, 1, total_tiles, max_m, lc, d_ops, d_coef, s, di)
                            : launch_fp32<true, 1, true>(d_entries, 1, total_tiles, max_m, lc, d_ops, d_coef, s, di);
    if (dt != SV_C64) return launch_fp32<true, 1, false>(d_entries, n_entries, total_tiles, max_m, 0, d_ops, d_coef, s, di);
    // two rows a thread while that fills the threads, else four (an amplitude loaded serves them all)
    if (max_m <= 11)
        return launch_fp32<false, 2, false>(d_entries, n_entries, total_tiles, max_m, 0, d_ops, d_coef, s, di);
    return launch_fp32<false, 4, false>(d_entries, n_entries, total_tiles, max_m, 0, d_ops, d_coef, s, di);
}

}  // namespace svk
