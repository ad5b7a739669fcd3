"""Plans of small states, which a batch shares: priced by what a batch of them
pays (the better of the general and the few-tile pass) and by its time alone, the
automatic plan is the best of all fusion widths; and a table that a caller installs is all that
the planner counts for its pair."""
import numpy as np
import pytest

from paper_2502_11385_gb300 import workloads as W
from test_lib_cpu import _table, sv  # noqa: F401  (fixture)

# ps per amplitude in a batch: pass, dense blocks of 1..5 qubits, diagonal, signs, permutations of 1..5
GENERAL = {"c64": (2.2, [0.8, 1.6, 3.5, 8.3, 15.9], 1.2, 1.5, [1.0, 1.3, 1.6, 3.0, 5.5]),
           "c128": (12.8, [3.2, 8.9, 16.0, 34.8, 113.0], 3.2, 3.0, [1.5, 2.1, 2.5, 5.0, 5.0])}
FEW = {"c64": (4.8, [1.4, 1.6, 2.3, 4.4, 8.7], 1.2, 1.2, [1.5, 1.6, 1.6, 1.6, 1.6]),
       "c128": (10.0, [4.2, 7.4, 14.0, 28.8, 59.0], 2.6, 1.9, [2.4, 2.6, 2.6, 2.6, 2.6])}


def _signs(v):
    return bool(np.all((v.imag == 0) & (np.abs(v.real) == 1)))


def _price(sv, p, table):  # noqa: F811
    a_pass, dense, diag, sign, perm = table
    s = p.summary()
    ps, ops = s["n_passes"] * a_pass, 0
    for i in range(s["n_blocks"]):
        ops += 1
        b = p.block(i)
        k, m = b["k"], b["mat"]
        if b["kind"] == sv.BLOCK_DIAG:
            ps += sign if _signs(m) else diag
        elif b["kind"] == sv.BLOCK_PERM:
            v = m[np.abs(m) > 0]
            quarter = bool(np.all(((v.imag == 0) & (np.abs(v.real) == 1)) | ((v.real == 0) & (np.abs(v.imag) == 1))))
            ps += perm[k - 1] + (0 if quarter else diag)
            ops += 0 if quarter else 1
        elif b["kind"] == sv.BLOCK_KRON:
            ps += k * dense[0]
            ops += k - 1
        else:
            ps += dense[k - 1]
    return ps, ops


def _circuits(n):
    yield "qaoa", W.qaoa(n, 2, n)[0]
    yield "hwea", W.hwea(n, 8, n)
    yield "brickwork", W.brickwork(n, 10, n)
    yield "aqft", W.aqft(n, 4)
    if n % 2 == 0:
        yield "adder", W.cuccaro_adder((n - 2) // 2)


@pytest.mark.parametrize("n", [6, 10, 12, 13, 14, 16, 17, 18])
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_plans_hold_for_batches(sv, dtype, n):  # noqa: F811
    """A plan's score weighs its time alone once and in a batch twice: a width that costs r
    times less in a batch takes r^2 times as long alone, or more.  (Alone, 0.6 us an op and
    4 us a pass, and the amplitudes of a CTA's share of a tile on every SM.)"""
    arith = sv.ARITH_NATIVE if dtype == "c64" else sv.ARITH_DF64
    m = min(n, 13 if dtype == "c64" else 12)
    share = max(0, min(3, 7 - (n - m), m - 8))

    def times(p):
        batch = [_price(sv, p, GENERAL[dtype])[0]] + ([_price(sv, p, FEW[dtype])[0]] if n >= 10 else [])
        ps, ops = _price(sv, p, FEW[dtype])
        return min(batch), ps * 1e-6 * max(2 ** n, 152 * 2 ** (m - share)) + 0.6 * ops + 4 * p.summary()["n_passes"]

    for name, g in _circuits(n):
        batch, alone = times(sv.Plan(n, dtype, g, sv.run_opts(arith=arith)))
        for k in range(1, 6):
            b, a = times(sv.Plan(n, dtype, g, sv.run_opts(arith=arith, max_fuse_k=k)))
            assert (batch / b) ** 2 <= a / alone * (1 + 1e-9), (name, k)


@pytest.mark.parametrize("n", [7, 12, 16, 20, 22])
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_an_installed_table_is_all_that_counts(sv, dtype, n):  # noqa: F811
    """The modelled time is the table's figures times the state's amplitudes and 4 us a
    launch, at every width: nothing of the built-in costs of states of few tiles is left."""
    arith = sv.ARITH_NATIVE if dtype == "c64" else sv.ARITH_DF64
    t = _table()
    table = (t["pass_ps"], t["dense_ps"][1:], t["diag_ps"], t["sign_ps"], t["perm_ps"][1:])
    try:
        sv.set_costs(dtype, arith, t)
        for _, g in _circuits(n):
            p = sv.Plan(n, dtype, g, sv.run_opts(arith=arith))
            want = _price(sv, p, table)[0] * 1e-9 * 2 ** n + 4e-3 * p.summary()["n_passes"]
            assert p.summary()["model_ms"] == pytest.approx(want, rel=1e-9)
    finally:
        sv.set_costs(dtype, arith, None)


@pytest.mark.parametrize("price", [float("inf"), float("nan"), 1e306])
@pytest.mark.parametrize("n", [7, 16, 22])
def test_blocks_priced_out_keep_their_gates(sv, n, price):  # noqa: F811
    """Wherever every width has a block that the table prices out, some plan is
    taken all the same, with every gate in it."""
    try:
        sv.set_costs("c64", sv.ARITH_NATIVE, _table(dense_ps=[0] + [price] * 5, diag_ps=price))
        for _, g in _circuits(n):
            assert sv.Plan(n, "c64", g, sv.run_opts(arith=sv.ARITH_NATIVE)).check() == 0
    finally:
        sv.set_costs("c64", sv.ARITH_NATIVE, None)
