"""The Builder's steps at their edges: marginals by warp sweeps (few and many
bins, whole and partial rows, distributions below a row, odd alignment) and the
contraction on the tensor cores and on the FP32 units, against the formula in
extended precision."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build_library()
    from paper_2502_11385_gb300 import sv as _sv
    return _sv


def _marginal(p, width, qubits):
    """Sums of the rows of p over every qubit not in `qubits`; bin bits in the order of `qubits`."""
    i = np.arange(1 << width)
    b = np.zeros_like(i)
    for j, q in enumerate(qubits):
        b |= ((i >> q) & 1) << j
    out = np.zeros((len(p), 1 << len(qubits)), dtype=np.longdouble)
    for v, row in enumerate(p):
        np.add.at(out[v], b, row.astype(np.longdouble))
    return out


def _terms(up, down, K, wa, cut_pos, wb, ka, kb):
    mu = _marginal(up, wa, ka + cut_pos).reshape(len(up), 1 << K, 1 << len(ka))
    md = _marginal(down, wb, kb)
    U, D = [], []
    for code in itertools.product(range(4), repeat=K):  # code[j]: term of cut j
        v = sum((0 if t <= 1 else t - 1) * 3 ** j for j, t in enumerate(code))
        u = np.zeros(1 << len(ka), dtype=np.longdouble)
        for y in range(1 << K):
            w = 1
            for j, t in enumerate(code):
                bit = (y >> j) & 1
                w *= (2 if bit == t else 0) if t <= 1 else 1 - 2 * bit
            u += w * mu[v][y]
        d = np.zeros(1 << len(kb), dtype=np.longdouble)
        rows = [(1, 0, 0, 0), (0, 1, 0, 0), (-1, -1, 2, 0), (-1, -1, 0, 2)]
        for s in itertools.product(range(4), repeat=K):
            w = np.prod([rows[t][x] for t, x in zip(code, s)])
            if w:
                d += int(w) * md[sum(x * 4 ** j for j, x in enumerate(s))]
        U.append(u)
        D.append(d)
    return np.array(U), np.array(D)


def _distributions(rng, count, width):
    p = rng.exponential(size=(count, 1 << width))
    p[:, :: 5] = 0.0
    p[:, 1:: 7] *= 2.0 ** -60
    p[0] = 0.0
    p[0, -1] = 1.0  # one outcome
    return p / p.sum(axis=1, keepdims=True)


@pytest.mark.parametrize("K,wa,wb,ka,kb", [
    (1, 2, 1, [0], [0]), (1, 5, 4, [0, 3], [1]), (1, 6, 6, [], []), (1, 7, 9, [6], [0, 8]),
    (2, 14, 17, [1], []), (1, 17, 6, [], [0, 1, 2, 3, 4, 5]), (2, 12, 13, list(range(10)), [2, 3, 5, 7, 11]),
    # the contraction on the tensor cores from 2^7 x 2^5 tiles and 2^20 outputs on, and just below
    (1, 9, 13, list(range(1, 8)), list(range(13))), (1, 9, 13, list(range(1, 7)), list(range(13))),
    (2, 17, 6, list(range(15)), list(range(5))), (3, 13, 11, list(range(10)), list(range(10))),
    (3, 11, 12, list(range(8)), list(range(12))), (4, 12, 10, list(range(8)), list(range(9)))])
def test_reconstruct_steps(sv, K, wa, wb, ka, kb):
    import torch
    rng = np.random.default_rng(100 * K + wa)
    cut_pos = [q for q in range(wa) if q not in ka][:K]
    up, down = _distributions(rng, 3 ** K, wa), _distributions(rng, 4 ** K, wb)
    U, D = _terms(up, down, K, wa, cut_pos, wb, ka, kb)
    want = (D.T @ U) / 2 ** K
    # 2^-53 on every term, and the products' digits or float pairs: 2^-46 of the columns' largest product a code
    tol = 2.0 ** -46 * 4 ** K / 2 ** K * np.abs(D).max(axis=0)[:, None] * np.abs(U).max(axis=0)[None, :] + 2.0 ** -100
    for shift in (0, 1):  # 16- and 8-byte aligned distributions
        def place(p):
            t = torch.zeros(p.size + shift, dtype=torch.float64, device="cuda")
            t[shift:] = torch.from_numpy(p.ravel())
            return list(t[shift:].view(p.shape))
        up_t, down_t = place(up), place(down)
        out = torch.full((want.size,), float("nan"), dtype=torch.float64, device="cuda")
        sv.cut_reconstruct(up_t, down_t, wa, cut_pos, wb, keep_mask_a=sum(1 << q for q in ka),
                           keep_mask_b=sum(1 << q for q in kb), out=out)
        got = out.cpu().numpy().reshape(want.shape)
        assert (np.abs(got - want.astype(np.float64)) <= tol.astype(np.float64)).all()
