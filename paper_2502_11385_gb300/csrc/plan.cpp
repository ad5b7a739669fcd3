// Host planner: gate matrices, fusion, tile-pass scheduling, cost model.
#include "plan.hpp"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace svp {

namespace {
inline int popc(uint64_t x) { return __builtin_popcountll(x); }
const double kPi = 3.14159265358979323846264338327950288;
}  // namespace

int gate_arity(int op) {
    if (op < 0 || op >= SV_NUM_OPS) return 0;
    return op >= SV_CX ? 2 : 1;
}

bool gate_is_diagonal(int op) {
    return op == SV_Z || op == SV_S || op == SV_T || op == SV_RZ || op == SV_CZ || op == SV_RZZ;
}

bool gate_is_monomial(int op) {
    return gate_is_diagonal(op) || op == SV_X || op == SV_Y || op == SV_CX || op == SV_SWAP;
}

void gate_matrix(const sv_gate& g, cd* m) {
    const cd I(0, 1);
    const int d = 1 << gate_arity(g.op);
    for (int i = 0; i < d * d; i++) m[i] = 0;
    double c = 0, s = 0;
    if (g.op == SV_RX || g.op == SV_RY || g.op == SV_U3) {
        c = std::cos(g.theta / 2);
        s = std::sin(g.theta / 2);
    }
    const double r2 = 1.0 / std::sqrt(2.0);
    auto ph = [](double a) { return cd(std::cos(a), std::sin(a)); };
    switch (g.op) {
        case SV_H: m[0] = r2; m[1] = r2; m[2] = r2; m[3] = -r2; break;
        case SV_X: m[1] = 1; m[2] = 1; break;
        case SV_Y: m[1] = -I; m[2] = I; break;
        case SV_Z: m[0] = 1; m[3] = -1; break;
        case SV_S: m[0] = 1; m[3] = I; break;
        case SV_T: m[0] = 1; m[3] = ph(kPi / 4); break;
        case SV_RX: m[0] = c; m[1] = -I * s; m[2] = -I * s; m[3] = c; break;
        case SV_RY: m[0] = c; m[1] = -s; m[2] = s; m[3] = c; break;
        case SV_RZ: m[0] = ph(-g.theta / 2); m[3] = ph(g.theta / 2); break;
        case SV_U3:
            m[0] = c;
            m[1] = -ph(g.lambda) * s;
            m[2] = ph(g.phi) * s;
            m[3] = ph(g.phi + g.lambda) * c;
            break;
        case SV_CX:  // local index b(q0) + 2 b(q1); flips b(q1) when b(q0) = 1
            for (int a = 0; a < 4; a++) {
                int b0 = a & 1, b1 = a >> 1;
                m[(b0 | ((b1 ^ b0) << 1)) * 4 + a] = 1;
            }
            break;
        case SV_CZ: m[0] = 1; m[5] = 1; m[10] = 1; m[15] = -1; break;
        case SV_RZZ: {
            cd a = ph(-g.theta / 2), b = ph(g.theta / 2);
            m[0] = a; m[5] = b; m[10] = b; m[15] = a;
            break;
        }
        case SV_SWAP:
            for (int a = 0; a < 4; a++) {
                int b0 = a & 1, b1 = a >> 1;
                m[(b1 | (b0 << 1)) * 4 + a] = 1;
            }
            break;
        default: break;
    }
}

int validate(int n, const sv_gate* g, size_t ng) {
    if (ng && !g) return SV_ERR_ARG;
    for (size_t t = 0; t < ng; t++) {
        int k = gate_arity(g[t].op);
        if (k == 0) return SV_ERR_ARG;
        if (!std::isfinite(g[t].theta) || !std::isfinite(g[t].phi) || !std::isfinite(g[t].lambda))
            return SV_ERR_ARG;
        if (g[t].q0 < 0 || g[t].q0 >= n) return SV_ERR_QUBIT;
        if (k == 2 && (g[t].q1 < 0 || g[t].q1 >= n || g[t].q1 == g[t].q0)) return SV_ERR_QUBIT;
    }
    return SV_OK;
}

static uint64_t gate_mask(const sv_gate& g) {
    uint64_t m = 1ull << g.q0;
    if (gate_arity(g.op) == 2) m |= 1ull << g.q1;
    return m;
}

// What fusion needs of a gate; a block has the flags that all its gates have.
enum GateFlag : uint8_t {
    GF_DIAG = 1,
    GF_MONO = 2,
    GF_ONEQ = 4,     // one-qubit
    GF_SIGN = 8,     // CZ or Z: signs only
    GF_QUARTER = 16  // no T, RZ, RZZ: phases of monomial gates are powers of i
};
struct GateInfo {
    uint64_t mask;
    int8_t q0, q1;  // q1 = q0 for one-qubit gates
    uint8_t flags;
};

static std::vector<GateInfo> gate_infos(const sv_gate* g, size_t ng) {
    std::vector<GateInfo> v(ng);
    for (size_t t = 0; t < ng; t++) {
        const int op = g[t].op;
        const bool one = gate_arity(op) == 1;
        v[t].mask = gate_mask(g[t]);
        v[t].q0 = (int8_t)g[t].q0;
        v[t].q1 = (int8_t)(one ? g[t].q0 : g[t].q1);
        v[t].flags = (uint8_t)((gate_is_diagonal(op) ? GF_DIAG : 0) | (gate_is_monomial(op) ? GF_MONO : 0) |
                               (one ? GF_ONEQ : 0) | (op == SV_CZ || op == SV_Z ? GF_SIGN : 0) |
                               (op != SV_T && op != SV_RZ && op != SV_RZZ ? GF_QUARTER : 0));
    }
    return v;
}

// A fusion before its matrices are formed: per block its qubits and flags, per
// gate its block.
struct Fusion {
    std::vector<uint64_t> mask;
    std::vector<uint8_t> flags;
    std::vector<int> block_of;
};

static int fused_kind(uint8_t flags, int k) {
    if (flags & GF_DIAG) return BK_DIAG;
    if (flags & GF_MONO) return BK_PERM;
    return (flags & GF_ONEQ) && k > 1 ? BK_KRON : BK_DENSE;
}

// Greedy fusion: each gate joins the latest block among those holding its
// qubits when the union stays within fuse_k qubits; otherwise it opens a new
// block.  fuse_k = 1 keeps every gate on its own.  keep_monomial = 1: a gate
// that is not monomial does not join a block made of monomial gates only (it
// opens a new block), so runs of X / CX / SWAP / diagonal gates stay
// permutation blocks; 2: a monomial gate does not join a block holding other
// gates either.  With pack, a gate that cannot join the latest block holding
// its qubits may join any later block with room, so gates on disjoint qubits
// share blocks (a layer of one-qubit gates becomes Kronecker blocks): the
// smallest of the last 64, the latest of these.  (No later block holds its
// qubits, so a block's room is all that counts: the last 64 blocks are kept as
// bits by size and kind, and a choice is a few bit operations.)
static void fuse(int n, const std::vector<GateInfo>& gi, int fuse_k, int keep_monomial, bool pack, Fusion& f) {
    const size_t ng = gi.size();
    f.mask.clear();
    f.flags.clear();
    f.mask.reserve(ng);
    f.flags.reserve(ng);
    f.block_of.resize(ng);
    int cur[64];
    std::fill(cur, cur + n, -1);  // latest block holding each qubit
    uint64_t open[kMaxFuse + 1][2] = {};  // bit b % 64: block b has that many qubits, and is monomial or not
    for (size_t t = 0; t < ng; t++) {
        const GateInfo& G = gi[t];
        const bool mono = G.flags & GF_MONO;
        const int bstar = std::max(cur[(int)G.q0], cur[(int)G.q1]);
        const bool not_mono_block = keep_monomial >= 1 && !mono, only_mono_block = keep_monomial >= 2 && mono;
        int target = -1;
        if (fuse_k > 1 && bstar >= 0) {
            const bool bm = f.flags[bstar] & GF_MONO;
            if (popc(f.mask[bstar] | G.mask) <= fuse_k && !(not_mono_block && bm) && !(only_mono_block && !bm))
                target = bstar;
        }
        const int nb = (int)f.mask.size();
        if (fuse_k > 1 && target < 0 && pack && nb - 1 > bstar) {
            const int newest = (nb - 1) & 63, depth = std::min(nb - 1 - bstar, 64);  // blocks that may take the gate
            const int arity = G.flags & GF_ONEQ ? 1 : 2;
            for (int k = 1; k + arity <= fuse_k && target < 0; k++) {
                uint64_t c = (not_mono_block ? 0 : open[k][1]) | (only_mono_block ? 0 : open[k][0]);
                c = newest == 63 ? c : (c << (63 - newest)) | (c >> (newest + 1));  // the newest block at bit 63
                if (depth < 64) c &= ~0ull << (64 - depth);
                if (c) target = nb - 1 - __builtin_clzll(c);
            }
        }
        if (target >= 0) {
            const uint64_t bit = 1ull << (target & 63);
            const bool recent = target > nb - 65;
            if (recent) open[popc(f.mask[target])][(f.flags[target] & GF_MONO) ? 1 : 0] &= ~bit;
            f.mask[target] |= G.mask;
            f.flags[target] &= G.flags;
            if (recent) open[popc(f.mask[target])][(f.flags[target] & GF_MONO) ? 1 : 0] |= bit;
        } else {
            target = nb;
            f.mask.push_back(G.mask);
            f.flags.push_back(G.flags);
            const uint64_t bit = 1ull << (nb & 63);
            for (auto& o : open) o[0] &= ~bit, o[1] &= ~bit;
            open[popc(G.mask)][mono ? 1 : 0] |= bit;
        }
        f.block_of[t] = target;
        cur[(int)G.q0] = cur[(int)G.q1] = target;
    }
}

// The blocks of a fusion, without matrices (sign_only and quarter are known
// from the gates: finalize() sets them from the entries).
static std::vector<Block> blocks_of(const Fusion& f) {
    std::vector<Block> blocks(f.mask.size());
    std::vector<int> count(blocks.size(), 0);
    for (int b : f.block_of) count[b]++;
    for (size_t b = 0; b < blocks.size(); b++) {
        Block& B = blocks[b];
        B.mask = f.mask[b];
        for (uint64_t left = B.mask; left; left &= left - 1) B.qubits[B.k++] = __builtin_ctzll(left);
        B.kind = fused_kind(f.flags[b], B.k);
        B.sign_only = B.kind == BK_DIAG && (f.flags[b] & GF_SIGN);
        B.quarter = B.kind == BK_PERM && (f.flags[b] & GF_QUARTER);
        B.gates.reserve(count[b]);
    }
    for (size_t t = 0; t < f.block_of.size(); t++) blocks[f.block_of[t]].gates.push_back((int)t);
    return blocks;
}

// Products of complex numbers by components: std::complex's own goes through a
// check for NaN (the gates are finite).
static inline cd mul(cd a, cd b) {
    return cd(a.real() * b.real() - a.imag() * b.imag(), a.real() * b.imag() + a.imag() * b.real());
}

namespace {
// Rows of a block's matrix under a gate: left-multiplication mixes the 2 or 4
// rows that differ in the gate's bits.
struct RowGate {
    int ga, gp[2], rows;  // qubits, block-local bits, rows mixed
    cd m[16];
    bool diag;
    int from[4];     // monomial gates: out row r = scale[r] * row from[r]
    cd scale[4];
};

RowGate row_gate(const Block& b, const sv_gate& g) {
    RowGate r;
    r.ga = gate_arity(g.op);
    r.gp[0] = r.gp[1] = 0;
    for (int j = 0; j < b.k; j++) {
        if (b.qubits[j] == g.q0) r.gp[0] = j;
        if (r.ga == 2 && b.qubits[j] == g.q1) r.gp[1] = j;
    }
    r.rows = 1 << r.ga;
    r.diag = gate_is_diagonal(g.op);
    gate_matrix(g, r.m);
    if (gate_is_monomial(g.op))
        for (int i = 0; i < r.rows; i++)
            for (int c = 0; c < r.rows; c++)
                if (r.m[i * r.rows + c] != cd(0, 0)) {
                    r.from[i] = c;
                    r.scale[i] = r.m[i * r.rows + c];
                }
    return r;
}

// The block rows that local row l of the gate stands for, in the group of r0.
inline int row_at(const RowGate& g, int r0, int l) {
    int r = r0 | (l & 1) << g.gp[0];
    if (g.ga == 2) r |= (l >> 1) << g.gp[1];
    return r;
}
inline int gate_bits(const RowGate& g) { return 1 << g.gp[0] | (g.ga == 2 ? 1 << g.gp[1] : 0); }
}  // namespace

void finalize(std::vector<Block>& blocks, const sv_gate* g, bool kron_mat) {
    constexpr int kD = 1 << kMaxFuse;
    double re[kD][kD], im[kD][kD];
    for (auto& b : blocks) {
        const int D = 1 << b.k;
        if (b.kind == BK_DIAG || b.kind == BK_PERM) {
            // a product of monomial gates: one nonzero per row, out[r] = phase[r] in[src[r]]
            int src[kD];
            cd phase[kD];
            for (int r = 0; r < D; r++) {
                src[r] = r;
                phase[r] = 1;
            }
            for (int t : b.gates) {
                const RowGate G = row_gate(b, g[t]);
                const int bits = gate_bits(G);
                for (int r0 = 0; r0 < D; r0++) {
                    if (r0 & bits) continue;
                    int s[4];
                    cd p[4];
                    for (int l = 0; l < G.rows; l++) {
                        const int from = row_at(G, r0, G.from[l]);
                        s[l] = src[from];
                        p[l] = mul(G.scale[l], phase[from]);
                    }
                    for (int l = 0; l < G.rows; l++) {
                        src[row_at(G, r0, l)] = s[l];
                        phase[row_at(G, r0, l)] = p[l];
                    }
                }
            }
            if (b.kind == BK_DIAG) {
                b.mat.assign(phase, phase + D);
                b.sign_only = true;
                for (const cd& v : b.mat)
                    b.sign_only = b.sign_only && v.imag() == 0.0 && std::fabs(v.real()) == 1.0;
                continue;
            }
            b.src.assign(src, src + D);
            b.phase.assign(phase, phase + D);
            b.quarter = true;
            for (const cd& v : b.phase)
                b.quarter = b.quarter && ((v.imag() == 0.0 && std::fabs(v.real()) == 1.0) ||
                                          (v.real() == 0.0 && std::fabs(v.imag()) == 1.0));
            continue;
        }
        if (b.kind == BK_KRON) {
            // per qubit, the product of its one-qubit gates in order
            b.factors.assign((size_t)4 * b.k, cd(0, 0));
            for (int j = 0; j < b.k; j++) b.factors[(size_t)4 * j] = b.factors[(size_t)4 * j + 3] = 1;
            for (int t : b.gates) {
                int j = 0;
                while (b.qubits[j] != g[t].q0) j++;
                cd u[4], *f = &b.factors[(size_t)4 * j];
                gate_matrix(g[t], u);
                const cd r[4] = {mul(u[0], f[0]) + mul(u[1], f[2]), mul(u[0], f[1]) + mul(u[1], f[3]),
                                 mul(u[2], f[0]) + mul(u[3], f[2]), mul(u[2], f[1]) + mul(u[3], f[3])};
                for (int e = 0; e < 4; e++) f[e] = r[e];
            }
            if (!kron_mat) continue;
        }
        for (int r = 0; r < D; r++)
            for (int c = 0; c < D; c++) {
                re[r][c] = r == c;
                im[r][c] = 0;
            }
        for (int t : b.gates) {
            const RowGate G = row_gate(b, g[t]);
            const int bits = gate_bits(G);
            for (int r0 = 0; r0 < D; r0++) {
                if (r0 & bits) continue;
                if (G.ga == 1 && !G.diag) {
                    const int r1 = r0 | bits;
                    const double a = G.m[0].real(), ai = G.m[0].imag(), c = G.m[1].real(), ci = G.m[1].imag();
                    const double d = G.m[2].real(), di = G.m[2].imag(), e = G.m[3].real(), ei = G.m[3].imag();
                    for (int j = 0; j < D; j++) {
                        const double x = re[r0][j], xi = im[r0][j], y = re[r1][j], yi = im[r1][j];
                        re[r0][j] = (a * x - ai * xi) + (c * y - ci * yi);
                        im[r0][j] = (a * xi + ai * x) + (c * yi + ci * y);
                        re[r1][j] = (d * x - di * xi) + (e * y - ei * yi);
                        im[r1][j] = (d * xi + di * x) + (e * yi + ei * y);
                    }
                    continue;
                }
                // every other gate is monomial: rows move and are scaled
                int order[4];
                for (int l = 0; l < G.rows; l++) order[l] = row_at(G, r0, l);
                double tr[4][kD], ti[4][kD];
                bool moved = false;
                for (int l = 0; l < G.rows; l++) moved = moved || G.from[l] != l;
                if (moved)
                    for (int l = 0; l < G.rows; l++)
                        for (int j = 0; j < D; j++) {
                            tr[l][j] = re[order[l]][j];
                            ti[l][j] = im[order[l]][j];
                        }
                for (int l = 0; l < G.rows; l++) {
                    const double sr = G.scale[l].real(), si = G.scale[l].imag();
                    const double* xr = moved ? tr[G.from[l]] : re[order[l]];
                    const double* xi = moved ? ti[G.from[l]] : im[order[l]];
                    if (G.from[l] == l && sr == 1.0 && si == 0.0) continue;
                    for (int j = 0; j < D; j++) {
                        const double x = xr[j], y = xi[j];
                        re[order[l]][j] = sr * x - si * y;
                        im[order[l]][j] = sr * y + si * x;
                    }
                }
            }
        }
        b.mat.resize((size_t)D * D);
        for (int r = 0; r < D; r++)
            for (int c = 0; c < D; c++) b.mat[(size_t)r * D + c] = cd(re[r][c], im[r][c]);
    }
}

std::vector<cd> block_matrix(const Block& b) {
    if (!b.mat.empty() || (b.kind != BK_PERM && b.kind != BK_KRON)) return b.mat;
    const int D = 1 << b.k;
    std::vector<cd> m((size_t)D * D, cd(0, 0));
    for (int r = 0; r < D; r++) {
        if (b.kind == BK_PERM) {
            m[(size_t)r * D + b.src[r]] = b.phase[r];
            continue;
        }
        for (int c = 0; c < D; c++) {
            cd v = 1;
            for (int j = 0; j < b.k; j++) v = mul(v, b.factors[(size_t)4 * j + ((r >> j) & 1) * 2 + ((c >> j) & 1)]);
            m[(size_t)r * D + c] = v;
        }
    }
    return m;
}

namespace {
// A block as the scheduler sees it.
struct SchedBlock {
    uint64_t mask;
    int index;
    int work;  // 2^k, 0 for a diagonal block (which joins any pass)
};
}  // namespace

// The blocks (in list order) that can run in one pass whose tile holds the
// qubits of `local`: a dense block joins when its qubits are local, a
// diagonal block always; a block that cannot join blocks its qubits for
// every later block of the pass (once all are blocked, none joins).  Returns
// the dense work joined (sum of 2^k); joins(i) for the blocks that join.
template <typename F>
static int64_t pass_with(const std::vector<SchedBlock>& todo, uint64_t all, uint64_t local, F joins) {
    uint64_t blocked = 0;
    int64_t work = 0;
    for (size_t i = 0; i < todo.size() && blocked != all; i++) {
        const SchedBlock& B = todo[i];
        if (!(B.mask & blocked) && (B.work == 0 || (B.mask & ~local) == 0)) {
            work += B.work;
            joins(i);
        } else {
            blocked |= B.mask;
        }
    }
    return work;
}

// Groups the blocks `todo` (in list order) into tile passes of tile_m qubits whose lowest
// `coalesce` qubits are always local (contiguous runs for coalesced loads); stops after
// `most` passes if blocks are left then.
static std::vector<Pass> schedule(int n, std::vector<SchedBlock>& todo, int tile_m, int coalesce, size_t most) {
    std::vector<Pass> passes;
    const size_t nb = todo.size();
    const uint64_t all = (n >= 64) ? ~0ull : ((1ull << n) - 1);
    if (tile_m >= n) {
        Pass p;
        p.local_mask = all;
        p.m = n;
        for (const SchedBlock& b : todo) p.blocks.push_back(b.index);
        if (nb) passes.push_back(p);
        todo.clear();
        return passes;
    }
    const int c = std::min(coalesce, n);
    const uint64_t low = (1ull << c) - 1;
    uint64_t used = 0;
    for (const SchedBlock& b : todo) used |= b.mask;
    auto fill = [&](uint64_t local) {  // up to tile_m qubits with the lowest unused ones
        for (int q = 0; q < n && popc(local) < tile_m; q++) local |= 1ull << q;
        return local;
    };
    std::vector<char> joined;
    while (!todo.empty() && passes.size() < most) {
        // candidate 1: greedy, the tile grows with the blocks in list order
        uint64_t local = low, blocked = 0;
        for (size_t i = 0; i < todo.size() && blocked != used; i++) {
            const SchedBlock& B = todo[i];
            if (B.mask & blocked) {
                blocked |= B.mask;
                continue;
            }
            if (B.work == 0) continue;
            const uint64_t need = local | B.mask;
            if (popc(need) <= tile_m) local = need;
            else blocked |= B.mask;
        }
        uint64_t best = fill(local);
        int64_t best_work = pass_with(todo, used, best, [](size_t) {});
        // candidates 2: the low qubits plus a contiguous window of the others
        const int w = tile_m - c;
        for (int s = c; w > 0 && s + w <= n; s++) {
            const uint64_t cand = low | (((1ull << w) - 1) << s);
            const int64_t work = pass_with(todo, used, cand, [](size_t) {});
            if (work > best_work) {
                best_work = work;
                best = cand;
            }
        }
        Pass p;
        joined.assign(todo.size(), 0);
        pass_with(todo, used, best, [&](size_t i) {
            joined[i] = 1;
            p.blocks.push_back(todo[i].index);
        });
        size_t left = 0;
        for (size_t i = 0; i < todo.size(); i++)
            if (!joined[i]) todo[left++] = todo[i];
        todo.resize(left);
        p.local_mask = best;
        p.m = popc(best);
        passes.push_back(std::move(p));
    }
    return passes;
}

static bool tc_arith(int arith) { return arith == AK_TC || arith == AK_TC32; }

static double block_flops(const Block& b, double dim, int arith) {
    // real flops (FMA = 2) of the block applied to the whole 2^n state
    if (b.kind == BK_DIAG) return b.sign_only ? 0.0 : 6.0 * dim;
    if (b.kind == BK_PERM) return b.quarter ? 0.0 : 6.0 * dim;  // moves, then a phase pass if not quarter
    if (b.kind == BK_KRON && !tc_arith(arith)) return 16.0 * (double)b.k * dim;  // k butterflies
    return 8.0 * (double)(1 << b.k) * dim;
}

// ALU lane instructions per amplitude for one block.
static double block_instr(const Block& b, int arith) {
    const double D = (double)(1 << b.k);
    const double cmac = arith == AK_DF64 ? 44.0 : 4.0;  // one complex multiply-add
    if (b.kind == BK_DIAG) {
        if (b.sign_only) return 1.0;
        return cmac;
    }
    if (b.kind == BK_PERM) return 2.0 + (b.quarter ? 0.0 : cmac);
    // complex multiply-add: 4 real FMAs; double-float: 4 x (TwoProd + cross
    // terms + TwoSum) = 44 FP32 instructions; a Kronecker block is k one-qubit
    // butterflies (2 multiply-adds per amplitude each)
    if (b.kind == BK_KRON) return cmac * 2.0 * b.k;
    return cmac * D;
}

// Tensor-core modes: 16-bit MMA flops per amplitude of a dense block (digit
// pairs of a real 2D x 2D product: 28 for complex128, 6 for the complex64
// triple split; blocks of fewer than 3 qubits padded to 3) and CUDA-core
// operations per amplitude (digit split, re-assembly).
static double tc_mma_flops(const Block& b, int arith) {
    if (b.kind == BK_DIAG || b.kind == BK_PERM) return 0.0;
    const int k = std::max(3, b.k);
    return (arith == AK_TC32 ? 6.0 : 28.0) * 8.0 * (double)(1 << k);
}
static double tc_alu(const Block& b, int arith) {
    if (b.kind == BK_DIAG) return b.sign_only ? 2.0 : (arith == AK_TC32 ? 4.0 : 40.0);
    if (b.kind == BK_PERM) return 4.0 + (b.quarter ? 0.0 : (arith == AK_TC32 ? 4.0 : 40.0));
    return arith == AK_TC32 ? 30.0 : 150.0;
}

// Measured cost of one block, picoseconds per amplitude (sv_costs).
static double measured_ps(const Block& b, int arith, const sv_costs& c) {
    const bool tc = tc_arith(arith);
    const int kd = tc ? std::max(3, b.k) : b.k;
    switch (b.kind) {
        case BK_DIAG: return b.sign_only ? c.sign_ps : c.diag_ps;
        case BK_PERM: return c.perm_ps[b.k] + (b.quarter ? 0.0 : c.diag_ps);
        case BK_KRON: return tc ? c.dense_ps[kd] : b.k * c.dense_ps[1];
        default: return c.dense_ps[kd];
    }
}

// Ops a tile runs for one block.
static int ops_of(const Block& b, int arith) {
    if (b.kind == BK_KRON && !tc_arith(arith)) return b.k;
    return b.kind == BK_PERM && !b.quarter ? 2 : 1;
}

// A plan's score from its time alone and its times in a batch, with weights 1 and 2 (of
// 95 batches and 127 circuits alone of 6 to 20 qubits: with equal weights three batches took
// 1.3 times as long as by plans for batches, with 1 and 3 six circuits alone lost 7 to 9 %
// of their time).
static double score(double alone, const double (&batch)[2], const Machine& mc) {
    if (!mc.batch[0]) return alone;
    const double b = (mc.batch[1] ? std::min(batch[0], batch[1]) : batch[0]) * mc.batch_states;
    return std::cbrt(alone * b * b);
}

// Time of one block from the measured costs.
static double measured_s(const Block& b, int arith, const Machine& mc, double dim) {
    return measured_ps(b, arith, *mc.measured) * 1e-12 * std::max(dim, mc.least_dim) + mc.op_s * ops_of(b, arith);
}

// Time of one block over the whole state, without the pass it joins: the
// measured table, else the analytic terms of model_cost for the block alone.
static double block_cost(const Block& b, int arith, const Machine& mc, double dim, int amp_bytes) {
    if (mc.measured) return measured_s(b, arith, mc, dim);
    const double rate = arith == AK_FP64 ? mc.fp64_ips : mc.fp32_ips;
    if (tc_arith(arith))
        return tc_alu(b, arith) * dim / rate +
               tc_mma_flops(b, arith) * dim / (arith == AK_TC32 ? mc.tc05_flops : mc.mma_flops);
    return std::max(block_instr(b, arith) * dim / rate, 2.0 * dim * amp_bytes / mc.smem_Bps);
}

double model_cost(const Plan& p, int amp_bytes, int arith, const Machine& mc, double* flops, double* alu_ops,
                  double* mma_flops) {
    const double dim = std::ldexp(1.0, p.n);
    const double state = dim * amp_bytes;
    const double rate = arith == AK_FP64 ? mc.fp64_ips : mc.fp32_ips;
    double total = 0, batch[2] = {0, 0}, fl_all = 0, ops_all = 0, mma_all = 0;
    for (const auto& ps : p.passes) {
        double fl = 0, instr = 0, smem = 0, mma = 0;
        for (int bi : ps.blocks) {
            fl += block_flops(p.blocks[bi], dim, arith);
            if (arith == AK_TC || arith == AK_TC32) {
                instr += tc_alu(p.blocks[bi], arith) * dim;
                mma += tc_mma_flops(p.blocks[bi], arith) * dim;
            } else {
                instr += block_instr(p.blocks[bi], arith) * dim;
            }
            smem += 2.0 * state;
        }
        if (arith == AK_DF64 || arith == AK_TC) instr += 60.0 * dim;  // float64 conversions per pass
        fl_all += fl;
        ops_all += instr;
        mma_all += mma;
        if (mc.measured) {  // a pass's measured time: its tile traffic plus each op's
            total += mc.measured->pass_ps * 1e-12 * std::max(dim, mc.least_dim) + mc.launch_s;
            for (int bi : ps.blocks) total += measured_s(p.blocks[bi], arith, mc, dim);
            for (int i = 0; i < 2 && mc.batch[i]; i++) {
                batch[i] += mc.batch[i]->pass_ps * 1e-12 * dim;
                for (int bi : ps.blocks) batch[i] += measured_ps(p.blocks[bi], arith, *mc.batch[i]) * 1e-12 * dim;
            }
            continue;
        }
        const double alu = instr / rate + mma / (arith == AK_TC32 ? mc.tc05_flops : mc.mma_flops);
        const double hbm = 2.0 * state / mc.hbm_Bps;
        const double sm = smem / mc.smem_Bps;
        total += std::max(std::max(alu, hbm), sm) + mc.launch_s;
    }
    if (flops) *flops = fl_all;
    if (alu_ops) *alu_ops = ops_all;
    if (mma_flops) *mma_flops = mma_all;
    return score(total, batch, mc);
}

Plan make_plan(int n, const sv_gate* g, size_t ng, int fuse_k, int tile_m, int coalesce,
               int amp_bytes, int arith, const Machine& mc) {
    Plan best;
    int k_lo = fuse_k > 0 ? fuse_k : 1, k_hi = fuse_k > 0 ? fuse_k : kMaxFuse;
    if (arith == AK_TC) {  // tensor-core blocks have at most 4 qubits
        k_hi = std::min(k_hi, 4);
        k_lo = std::min(k_lo, k_hi);
    }
    // the tensor-core modes pad blocks below 3 qubits to 3, so narrower
    // fusion only adds blocks: the autotuner starts at 3 there
    if (fuse_k == 0 && tc_arith(arith)) k_lo = std::min(3, k_hi);
    // the autotuner: every fusion width, with and without keeping runs of
    // monomial gates as permutation blocks, with and without packing gates
    // on disjoint qubits into one block.  The variants of a width are scored
    // by their blocks' cost alone and only the cheapest is scheduled into
    // passes, then the widths are compared by the full cost model.  With measured
    // costs a plan's time is its blocks' plus its passes', so the candidates are
    // scheduled from the cheapest blocks on and not at all once the blocks and
    // one pass cost more than the best plan.  For states of few tiles (Machine::batch)
    // every variant of a width is a candidate: there the passes are many of a plan's
    // costs (17 qubits complex64 QAOA: the variant of the cheapest blocks took 102 ps an
    // amplitude of a batch, one of dearer blocks and other passes 79).
    const double dim = std::ldexp(1.0, n);
    const std::vector<GateInfo> gi = gate_infos(g, ng);
    bool any_mono = false, any_other = false;
    for (const GateInfo& x : gi) (x.flags & GF_MONO ? any_mono : any_other) = true;
    // cost of a block by its size and flags, alone and in a batch
    double cost_of[kMaxFuse + 1][32], batch_of[kMaxFuse + 1][32][2] = {};
    for (int k = 1; k <= kMaxFuse; k++)
        for (int fl = 0; fl < 32; fl++) {
            Block b;
            b.k = k;
            b.kind = fused_kind((uint8_t)fl, k);
            b.sign_only = fl & GF_SIGN;
            b.quarter = fl & GF_QUARTER;
            cost_of[k][fl] = block_cost(b, arith, mc, dim, amp_bytes);
            for (int i = 0; i < 2 && mc.batch[i]; i++)
                batch_of[k][fl][i] = measured_ps(b, arith, *mc.batch[i]) * 1e-12 * dim;
        }
    const double pass_s =
        mc.measured ? mc.measured->pass_ps * 1e-12 * std::max(dim, mc.least_dim) + mc.launch_s : -1e300;
    auto plan_s = [&](double cost, const double (&batch)[2], double passes) {  // of blocks of this cost in so many passes
        double b[2];
        for (int i = 0; i < 2; i++) b[i] = mc.batch[i] ? batch[i] + passes * mc.batch[i]->pass_ps * 1e-12 * dim : 0;
        return score(cost + passes * pass_s, b, mc);
    };
    struct Candidate {
        int k = 0;
        double cost = 0, batch[2] = {0, 0};  // of its blocks
        double least = 0;                    // of any plan of it: with one pass
        Fusion f;
    };
    constexpr double kTie = 1e-13;  // sums of the same costs in another order
    constexpr double kMost = 1e300;
    const bool one_pass = mc.measured && n <= tile_m;
    std::vector<Candidate> cands;
    Fusion f;
    for (int k = k_lo; k <= k_hi; k++) {
        const size_t first = cands.size();
        for (int variant = 0; variant < (k > 1 ? 6 : 1); variant++) {
            if (variant % 3 > 0 && !(any_mono && any_other)) continue;  // the same blocks as keep_monomial = 0
            fuse(n, gi, k, variant % 3, variant >= 3, f);
            double cost = 0, batch[2] = {0, 0};
            for (size_t b = 0; b < f.mask.size(); b++) {
                const int bk = popc(f.mask[b]), fl = f.flags[b];
                cost += cost_of[bk][fl];
                for (int i = 0; i < 2; i++) batch[i] += batch_of[bk][fl][i];
            }
            // one candidate of all (a plan of one pass has its score already), every variant, or one
            // a width; at the same cost (a Kronecker block outside the tensor-core modes is its
            // butterflies), fewer blocks
            double least = plan_s(cost, batch, 1);
            if (!(least < kMost)) least = kMost;  // (an installed table may price blocks out with infinity)
            if (one_pass) {
                if (cands.empty()) cands.emplace_back();
            } else if (mc.batch[0]) {
                bool again = false;  // the same blocks as another variant's
                for (size_t i = first; i < cands.size() && !again; i++)
                    again = cands[i].f.mask == f.mask && cands[i].f.flags == f.flags;
                if (again) continue;
                cands.emplace_back();
            } else if (cands.size() == first) {
                cands.emplace_back();
            }
            Candidate& c = cands.back();
            const double now = mc.batch[0] || one_pass ? least : cost, was = mc.batch[0] || one_pass ? c.least : c.cost;
            const double tie = one_pass ? kTie : 1e-9;
            if (c.k == 0 || now < was * (1 - tie) || (now < was * (1 + tie) && f.mask.size() < c.f.mask.size())) {
                c.k = k;
                c.cost = cost;
                std::copy(batch, batch + 2, c.batch);
                c.least = least;
                std::swap(c.f, f);
            }
        }
    }
    if (mc.measured)
        std::stable_sort(cands.begin(), cands.end(),
                         [](const Candidate& a, const Candidate& b) { return a.least < b.least; });
    const Candidate* chosen = nullptr;
    double chosen_s = kMost;
    std::vector<SchedBlock> todo;
    for (const Candidate& c : cands) {
        if (c.least > chosen_s * (1 + kTie)) continue;
        todo.resize(c.f.mask.size());
        for (size_t b = 0; b < todo.size(); b++) {
            const int k = popc(c.f.mask[b]);
            todo[b] = {c.f.mask[b], (int)b, fused_kind(c.f.flags[b], k) == BK_DIAG ? 0 : 1 << k};
        }
        size_t most = todo.size();  // passes, of a plan that may be chosen
        if (mc.measured && chosen) {
            most = 1;
            while (most < todo.size() && plan_s(c.cost, c.batch, (double)(most + 1)) <= chosen_s * (1 + kTie)) most++;
        }
        std::vector<Pass> passes = schedule(n, todo, std::min(tile_m, n), std::min(coalesce, n), most);
        if (!todo.empty()) continue;
        double s;
        if (mc.measured) {
            s = plan_s(c.cost, c.batch, (double)passes.size());
        } else {
            Plan p;
            p.n = n;
            p.blocks = blocks_of(c.f);
            p.passes = passes;
            s = model_cost(p, amp_bytes, arith, mc, nullptr);
        }
        if (!chosen || s < chosen_s * (1 - kTie) || (s < chosen_s * (1 + kTie) && c.f.mask.size() < chosen->f.mask.size())) {
            chosen = &c;
            chosen_s = s;
            best.passes.swap(passes);
        }
    }
    best.n = n;
    best.fuse_k = chosen->k;
    best.tile_m = std::min(tile_m, n);
    best.coalesce = std::min(coalesce, n);
    best.blocks = blocks_of(chosen->f);
    finalize(best.blocks, g, tc_arith(arith));
    double fl = 0, ops = 0, mma = 0;
    best.model_s = model_cost(best, amp_bytes, arith, mc, &fl, &ops, &mma);
    best.flops = fl;
    best.alu_ops = ops;
    best.mma_flops = mma;
    return best;
}

int check_plan(const Plan& p, size_t ng, const sv_gate* g) {
    std::vector<int> seen(ng, 0);
    std::vector<int> last(p.n, -1);  // last gate index applied per qubit
    std::vector<char> used(p.blocks.size(), 0);
    for (const auto& ps : p.passes) {
        if (popc(ps.local_mask) != ps.m) return 1;
        for (int bi : ps.blocks) {
            if (bi < 0 || bi >= (int)p.blocks.size() || used[bi]) return 2;
            used[bi] = 1;
            const Block& b = p.blocks[bi];
            if (b.k < 1 || b.k > kMaxFuse) return 3;
            if (b.kind != BK_DIAG && (b.mask & ~ps.local_mask)) return 4;
            for (int t : b.gates) {
                if (t < 0 || (size_t)t >= ng || seen[t]) return 5;
                seen[t] = 1;
                uint64_t gm = gate_mask(g[t]);
                if (gm & ~b.mask) return 6;
                for (int q = 0; q < p.n; q++) {
                    if (!((gm >> q) & 1)) continue;
                    if (last[q] > t) return 7;  // per-qubit order broken
                    last[q] = t;
                }
            }
        }
    }
    for (size_t t = 0; t < ng; t++)
        if (!seen[t]) return 8;
    return 0;
}

}  // namespace svp
