"""Cases that a user of the statevector engine runs, each through the package's
public entry points (paper_2502_11385_gb300.sv).

Four kinds of work, the ones the package is for:

``circuit``      one circuit on a state handle that the program keeps: reset,
                 apply_circuit, then the result: the probabilities beside the
                 statevector (complex128), or the statevector (complex64).
``batch``        the CutQC Evaluator's subcircuit instances, prepared once and
                 executed for their probability vectors.
``reconstruct``  the CutQC Builder: variant distributions to the distribution of
                 the uncut circuit over chosen qubits.
``readout``      a simulated state to its probabilities, a marginal over chosen qubits and
                 its norm.

Widths are qubit counts, so a step of one doubles the work; circuits come from
paper_2502_11385_gb300.workloads with angles, graphs and inputs of the seed.
"""
import math
import random

import numpy as np
import torch

from paper_2502_11385_gb300 import sv, workloads as W

DEV = "cuda"
TORCH_DTYPE = {"c64": torch.complex64, "c128": torch.complex128}
# gate applications x amplitudes of the largest listed case (30 qubits, 920 gates)
MOST_WORK = 920 << 30


def listed():
    return [
        # the smallest request of a serving stream: all latency, the statevector read on the host
        {"name": "qaoa_10q_c64_host", "kind": "circuit", "family": "qaoa", "n": 10, "depth": 2, "dtype": "c64",
         "out": "host"},
        # the 12-qubit brickwork of the oracle tests, probabilities into a numpy array
        {"name": "brickwork_12q_c128_host", "kind": "circuit", "family": "brickwork", "n": 12, "depth": 10,
         "dtype": "c128", "out": "host"},
        # a variational ansatz at the width such loops run at, complex128
        {"name": "hwea_17q_c128", "kind": "circuit", "family": "hwea", "n": 17, "depth": 8, "dtype": "c128",
         "out": "device"},
        # an upstream subcircuit of the 40-qubit cut on its own, in single precision
        {"name": "brickwork_21q_c64", "kind": "circuit", "family": "brickwork", "n": 21, "depth": 12, "dtype": "c64",
         "out": "device"},
        # QAOA on a 3-regular graph (odd width: one vertex of lower degree): many diagonal two-qubit gates
        {"name": "qaoa_23q_c128", "kind": "circuit", "family": "qaoa", "n": 23, "depth": 2, "dtype": "c128",
         "out": "device"},
        # the ripple-carry adder on superposed registers: mostly CX, T and H
        {"name": "adder_26q_c128", "kind": "circuit", "family": "adder", "n": 26, "depth": 1, "dtype": "c128",
         "out": "device"},
        # the approximate Fourier transform of a basis state: controlled phases
        {"name": "aqft_27q_c64", "kind": "circuit", "family": "aqft", "n": 27, "depth": 5, "dtype": "c64",
         "out": "device"},
        # the benchmark's circuit in single precision, one qubit below its width
        {"name": "ghz_brickwork_29q_c64", "kind": "circuit", "family": "ghz_brickwork", "n": 29, "depth": 20,
         "dtype": "c64", "out": "device"},
        # the benchmark's circuit: 30 qubits, complex128, 920 gates
        {"name": "ghz_brickwork_30q_c128", "kind": "circuit", "family": "ghz_brickwork", "n": 30, "depth": 20,
         "dtype": "c128", "out": "device"},
        # the Evaluator's 91 instances of the 40-qubit circuit cut at three wires into 21 + 22 qubits
        {"name": "cut40_batch_c128", "kind": "batch", "width_a": 21, "width_b": 22, "cuts": 3, "depth": 12,
         "dtype": "c128"},
        # the Builder on the same cut: 12 + 12 chosen qubits
        {"name": "cut40_reconstruct", "kind": "reconstruct", "width_a": 21, "width_b": 22, "cuts": 3, "keep_a": 12,
         "keep_b": 12},
        # reading a simulated state: all probabilities, a marginal over 10 qubits, the norm
        {"name": "readout_28q_c64", "kind": "readout", "n": 28, "keep": 10, "dtype": "c64"},
    ]


def draw(rng):
    kind = rng.choice(["circuit"] * 7 + ["batch", "reconstruct", "readout"])
    if kind == "circuit":
        n = rng.randint(10, 30)
        family = rng.choice(["brickwork", "ghz_brickwork", "qaoa", "hwea", "aqft", "adder", "supremacy"])
        depth = {"brickwork": rng.randint(5, 40), "ghz_brickwork": rng.randint(5, 25), "qaoa": rng.randint(1, 4),
                 "hwea": rng.randint(2, 12), "aqft": rng.randint(2, 6), "adder": 1,
                 "supremacy": rng.randint(8, 24)}[family]
        if family == "adder":
            n -= n % 2  # two registers, a carry in and a carry out
        if family == "supremacy":
            n = max(12, n)
        case = {"kind": kind, "family": family, "n": n, "depth": depth, "dtype": rng.choice(["c64", "c128"]),
                "out": "host" if n <= 14 and rng.random() < 0.5 else "device"}
        while case["depth"] > 1 and len(_gates(case, 0)[0]) << _qubits(case) > MOST_WORK * 3 // 4:
            case["depth"] -= 1
        return case
    if kind == "batch":
        cuts = rng.randint(1, 3)
        return {"kind": kind, "width_a": rng.randint(10, 21), "width_b": rng.randint(10, 21), "cuts": cuts,
                "depth": 2 * rng.randint(3, 6), "dtype": "c128"}
    if kind == "reconstruct":
        cuts = rng.randint(1, 4)
        wa, wb = rng.randint(10, 21), rng.randint(10, 21)
        return {"kind": kind, "width_a": wa, "width_b": wb, "cuts": cuts,
                "keep_a": rng.randint(4, min(12, wa - cuts)), "keep_b": rng.randint(4, min(12, wb))}
    return {"kind": kind, "n": rng.randint(14, 29), "keep": rng.randint(1, 14), "dtype": rng.choice(["c64", "c128"])}


# --------------------------------------------------------------------------
# Inputs of a case.
# --------------------------------------------------------------------------
def _qubits(case):
    if case["family"] == "supremacy":
        rows = max(2, int(math.sqrt(case["n"])))
        return rows * (case["n"] // rows)
    return case["n"]


def _gates(case, seed):
    """(gate list, initial basis state) of a circuit case."""
    n, depth, rng = _qubits(case), case["depth"], random.Random(seed)
    family = case["family"]
    if family == "brickwork":
        return W.brickwork(n, depth, seed), 0
    if family == "ghz_brickwork":
        return W.concat(W.ghz_prefix(n), W.brickwork(n, depth, seed)), 0
    if family == "qaoa":
        return W.qaoa(n, depth, seed)[0], 0
    if family == "hwea":
        return W.hwea(n, depth, seed), 0
    if family == "aqft":
        return W.aqft(n, depth), rng.randrange(1 << n)
    if family == "adder":
        registers = W.gates([(W.RY, q, -1, math.pi * rng.random()) for q in range(1, n - 1)])
        return W.concat(registers, W.cuccaro_adder((n - 2) // 2)), 0
    rows = max(2, int(math.sqrt(case["n"])))
    return W.supremacy(rows, n // rows, depth, seed), 0


def _cut(case, seed):
    n = case["width_a"] + case["width_b"] - case["cuts"]
    return W.cuttable_brickwork(n, case["depth"], seed, cut_lo=case["width_a"] - case["cuts"], n_cuts=case["cuts"],
                                switch_layer=case["depth"] // 2)


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _distributions(count, width, gen):
    """Distributions as random circuits give them: exponential weights, summing to one."""
    p = torch.empty((count, 1 << width), dtype=torch.float64, device=DEV).exponential_(generator=gen)
    return p.div_(p.sum(dim=1, keepdim=True))


def _reconstruct_inputs(case, seed):
    gen, rng = _generator(seed), random.Random(seed)
    wa, wb, cuts = case["width_a"], case["width_b"], case["cuts"]
    cut_pos = list(range(wa - cuts, wa))
    keep_a = sum(1 << q for q in rng.sample(range(wa - cuts), case["keep_a"]))
    keep_b = sum(1 << q for q in rng.sample(range(wb), case["keep_b"]))
    return _distributions(3 ** cuts, wa, gen), _distributions(4 ** cuts, wb, gen), cut_pos, keep_a, keep_b


def _readout_inputs(case, seed):
    """A normalised state with the amplitudes of a random circuit, and the mask of the marginal."""
    a = torch.randn(1 << case["n"], dtype=TORCH_DTYPE[case["dtype"]], device=DEV, generator=_generator(seed))
    a.div_(torch.linalg.vector_norm(torch.view_as_real(a), dtype=torch.float64).item())
    qubits = random.Random(seed).sample(range(case["n"]), case["keep"])
    return a, sum(1 << q for q in qubits)


def prepare(case, seed):
    st = {"case": case}
    if case["kind"] == "circuit":
        st["gates"], st["basis"] = _gates(case, seed)
        n = _qubits(case)
        if case["out"] == "host":
            st["state"] = sv.create(n, case["dtype"])
            return st
        st["amp"] = torch.empty(1 << n, dtype=TORCH_DTYPE[case["dtype"]], device=DEV)
        st["state"] = sv.State.from_tensor(st["amp"], n, case["dtype"])
        if case["dtype"] == "c128":
            st["p"] = torch.empty(1 << n, dtype=torch.float64, device=DEV)
    elif case["kind"] == "batch":
        cc = _cut(case, seed)
        st["up"] = torch.empty((3 ** cc.n_cuts, 1 << cc.width_a), dtype=torch.float64, device=DEV)
        st["down"] = torch.empty((4 ** cc.n_cuts, 1 << cc.width_b), dtype=torch.float64, device=DEV)
        items = [(cc.width_a, case["dtype"], g, o) for g, o in zip(cc.upstream_variants(), st["up"])]
        items += [(cc.width_b, case["dtype"], g, o) for g, o in zip(cc.downstream_variants(), st["down"])]
        st["batch"] = sv.Batch(items)
    elif case["kind"] == "reconstruct":
        up, down, st["cut_pos"], st["keep_a"], st["keep_b"] = _reconstruct_inputs(case, seed)
        st["up"], st["down"] = list(up), list(down)
        st["p"] = torch.empty(1 << (case["keep_a"] + case["keep_b"]), dtype=torch.float64, device=DEV)
    else:
        st["amp"], st["mask"] = _readout_inputs(case, seed)
        st["state"] = sv.State.from_tensor(st["amp"], case["n"], case["dtype"])
        st["p"] = torch.empty(1 << case["n"], dtype=torch.float64, device=DEV)
        st["m"] = torch.empty(1 << case["keep"], dtype=torch.float64, device=DEV)
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "circuit":
        s = st["state"]
        s.reset(st["basis"])
        s.apply_circuit(st["gates"])
        if case["out"] == "host":
            return s.probabilities() if case["dtype"] == "c128" else s.amplitudes()
        if case["dtype"] == "c128":
            return {"statevector": st["amp"], "probabilities": s.probabilities(st["p"])}
        return st["amp"]
    if case["kind"] == "batch":
        st["batch"].execute()
        return {"up": st["up"], "down": st["down"]}
    if case["kind"] == "reconstruct":
        return sv.cut_reconstruct(st["up"], st["down"], case["width_a"], st["cut_pos"], case["width_b"],
                                  keep_mask_a=st["keep_a"], keep_mask_b=st["keep_b"], out=st["p"])
    s = st["state"]
    return {"probabilities": s.probabilities(st["p"]), "marginal": s.marginal_probabilities(st["mask"], st["m"]),
            "norm": s.norm()}


def work(case):
    amp = 8 if case.get("dtype") == "c64" else 16
    if case["kind"] == "circuit":
        # the result written once (the initial state is a basis index); every gate's products
        dim = 1 << _qubits(case)
        out = amp if case["dtype"] == "c64" else (8 if case["out"] == "host" else amp + 8)
        return {"bytes": dim * out, "flops": dim * _gate_flops(_gates(case, 0)[0])}
    if case["kind"] == "batch":
        cc = _cut(case, 0)
        b = f = 0
        for width, variants in ((cc.width_a, cc.upstream_variants()), (cc.width_b, cc.downstream_variants())):
            b += len(variants) * 8 << width
            f += sum(_gate_flops(g) for g in variants) << width
        return {"bytes": b, "flops": f}
    if case["kind"] == "reconstruct":
        variants = (3 ** case["cuts"] << case["width_a"]) + (4 ** case["cuts"] << case["width_b"])
        outs = 1 << (case["keep_a"] + case["keep_b"])
        return {"bytes": 8 * (variants + outs), "flops": variants + outs * 2 * 4 ** case["cuts"]}
    # the state read once for all three results
    dim = 1 << case["n"]
    return {"bytes": dim * (amp + 8) + (8 << case["keep"]), "flops": 5 * dim}


def _gate_flops(gates):
    """Real flops per amplitude, gate by gate: 14 for a 2 x 2 product, 6 for a phase, none for a move or a sign."""
    per = {W.H: 14, W.RX: 14, W.RY: 14, W.U3: 14, W.S: 3, W.T: 3, W.RZ: 6, W.RZZ: 6}
    return sum(per.get(int(op), 0) for op in gates["op"])


# --------------------------------------------------------------------------
# The same results in 64 bits, from torch alone.
# --------------------------------------------------------------------------
def _matrix(g):
    """2 x 2 matrix (rows) of a one-qubit gate, Qiskit's conventions."""
    op, t, p, l = int(g["op"]), float(g["theta"]), float(g["phi"]), float(g["lam"])
    c, s, r = math.cos(t / 2), math.sin(t / 2), math.sqrt(0.5)
    e = lambda x: complex(math.cos(x), math.sin(x))
    return {W.H: ((r, r), (r, -r)), W.X: ((0, 1), (1, 0)), W.Y: ((0, -1j), (1j, 0)), W.Z: ((1, 0), (0, -1)),
            W.S: ((1, 0), (0, 1j)), W.T: ((1, 0), (0, e(math.pi / 4))), W.RX: ((c, -1j * s), (-1j * s, c)),
            W.RY: ((c, -s), (s, c)), W.RZ: ((e(-t / 2), 0), (0, e(t / 2))),
            W.U3: ((c, -e(l) * s), (e(p) * s, e(p + l) * c))}[op]


def _simulate(n, gates, basis):
    """The statevector, gate by gate, in complex128."""
    a = torch.zeros(1 << n, dtype=torch.complex128, device=DEV)
    a[basis] = 1
    for g in gates:
        op, q0, q1 = int(g["op"]), int(g["q0"]), int(g["q1"])
        if op not in W.TWO_QUBIT:
            v = a.view(-1, 2, 1 << q0)
            x, y, (m0, m1) = v[:, 0], v[:, 1], _matrix(g)
            if m0[1] == 0 and m1[0] == 0:
                for part, u in ((x, m0[0]), (y, m1[1])):
                    if u != 1:
                        part.mul_(u)
                continue
            old = x.clone()
            x.mul_(m0[0]).add_(y, alpha=m0[1])
            y.mul_(m1[1]).add_(old, alpha=m1[0])
            continue
        hi, lo = max(q0, q1), min(q0, q1)
        v = a.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
        at = lambda b0, b1: v[:, b0 if q0 == hi else b1, :, b1 if q0 == hi else b0]
        if op == W.CZ:
            at(1, 1).neg_()
        elif op == W.RZZ:
            t = float(g["theta"]) / 2
            for b0 in (0, 1):
                for b1 in (0, 1):
                    at(b0, b1).mul_(complex(math.cos(t), math.sin(t) if b0 != b1 else -math.sin(t)))
        else:
            x, y = (at(1, 0), at(1, 1)) if op == W.CX else (at(1, 0), at(0, 1))
            old = x.clone()
            x.copy_(y)
            y.copy_(old)
    return a


def _probs(a):
    return a.real.double().square() + a.imag.double().square()


def _marginal(p, width, qubits):
    """Sum over every qubit but `qubits` along the last axis; index bits in ascending qubit order."""
    for q in reversed(range(width)):
        if q not in qubits:
            p = p.reshape(*p.shape[:-1], -1, 2, 1 << q).sum(dim=-2).flatten(-2)
    return p


def exact(case, seed):
    if case["kind"] == "circuit":
        n = _qubits(case)
        gates, basis = _gates(case, seed)
        if len(gates) << n > 900 << 29:
            return None  # takes over 20 seconds
        a = _simulate(n, gates, basis)
        if case["dtype"] == "c64":
            return a.cpu().numpy() if case["out"] == "host" else a
        p = _probs(a)
        return p.cpu().numpy() if case["out"] == "host" else {"statevector": a, "probabilities": p}
    if case["kind"] == "batch":
        cc = _cut(case, seed)
        variants = cc.upstream_variants(), cc.downstream_variants()
        if sum(len(g) << w for w, gs in zip((cc.width_a, cc.width_b), variants) for g in gs) > 900 << 29:
            return None
        return {key: torch.stack([_probs(_simulate(w, g, 0)) for g in gs])
                for key, w, gs in (("up", cc.width_a, variants[0]), ("down", cc.width_b, variants[1]))}
    if case["kind"] == "reconstruct":
        return _reconstruct(case, seed)
    a, mask = _readout_inputs(case, seed)
    p = _probs(a)
    kept = [q for q in range(case["n"]) if mask >> q & 1]
    return {"probabilities": p, "marginal": _marginal(p, case["n"], kept), "norm": float(p.sum())}


def _reconstruct(case, seed):
    """2^-K sum_i U_i D_i over the terms i of every cut (I/Z with outcome 0 and 1, X, Y; |0>, |1>, 2|+> - |0> - |1>,
    2|+i> - |0> - |1>)."""
    up, down, cut_pos, keep_a, keep_b = _reconstruct_inputs(case, seed)
    wa, wb, cuts = case["width_a"], case["width_b"], case["cuts"]
    u = _marginal(up, wa, [q for q in range(wa) if keep_a >> q & 1] + cut_pos)  # cut qubits: the highest bits
    d = _marginal(down, wb, [q for q in range(wb) if keep_b >> q & 1])
    na, nb = 1 << case["keep_a"], 1 << case["keep_b"]
    # term of one cut from (basis, outcome), and from the initial state
    tu = torch.zeros((4, 3, 2), dtype=torch.float64, device=DEV)
    tu[0, 0, 0] = tu[1, 0, 1] = 2
    tu[2, 1, 0], tu[2, 1, 1], tu[3, 2, 0], tu[3, 2, 1] = 1, -1, 1, -1
    td = torch.tensor([[1, 0, 0, 0], [0, 1, 0, 0], [-1, -1, 2, 0], [-1, -1, 0, 2]], dtype=torch.float64, device=DEV)
    u = u.reshape(*[3] * cuts, *[2] * cuts, na)  # axes: bases of cuts K-1..0, outcomes of cuts K-1..0
    d = d.reshape(*[4] * cuts, nb)
    for j in range(cuts):  # the last basis axis is the lowest cut's; each turn adds a term axis at the front
        u = torch.tensordot(tu, u, dims=([1, 2], [cuts - 1, 2 * cuts - 1 - j]))
        d = torch.tensordot(td, d, dims=([1], [cuts - 1]))
    u, d = u.reshape(-1, na), d.reshape(-1, nb)
    return (d.T @ u).reshape(-1) / (1 << cuts)
