"""The planner's search: the automatic plan costs no more than the plan of any
single fusion width (widths that cannot win are skipped, none that can), and
the greedy fusion keeps every gate's order with more than 64 blocks open."""
import numpy as np
import pytest

import oracle
from paper_2502_11385_gb300 import workloads as W
from test_lib_cpu import _plan_unitary_state, sv  # noqa: F401  (fixture)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,g", [
    (9, W.brickwork(9, 8, 1)), (14, W.qaoa(14, 2, 2)[0]), (20, W.hwea(20, 3, 3)), (24, W.aqft(24, 4)),
    (26, W.cuccaro_adder(12)), (30, W.gates([(W.H, q, -1) for q in range(30)])), (30, W.gates([(W.T, 0, -1)]))])
def test_search_is_exact(sv, n, g, dtype):  # noqa: F811
    for arith in (sv.ARITH_AUTO, sv.ARITH_NATIVE, sv.ARITH_TC):
        auto = sv.Plan(n, dtype, g, sv.run_opts(arith=arith))
        assert auto.check() == 0
        costs = []
        tc = arith == sv.ARITH_TC or (arith == sv.ARITH_AUTO and n >= (23 if dtype == "c64" else 20))
        for k in range(3 if tc else 1, 6):  # the tensor-core modes pad narrower blocks to 3 qubits
            p = sv.Plan(n, dtype, g, sv.run_opts(arith=arith, max_fuse_k=k))
            assert p.check() == 0
            costs.append(p.summary()["model_ms"])
        assert auto.summary()["model_ms"] == pytest.approx(min(costs), rel=1e-12)


def test_packing_over_many_blocks(sv):  # noqa: F811
    n = 7
    rng = np.random.default_rng(11)
    rows = []
    for _ in range(100):
        q = rng.permutation(n)
        rows.append((int(rng.choice([W.CX, W.CZ, W.RZZ, W.SWAP])), int(q[0]), int(q[1]), float(rng.uniform(-3, 3))))
        rows.append((int(rng.choice([W.U3, W.H, W.T, W.X])), int(q[2]), -1, *rng.uniform(-3, 3, 3)))
    g = W.gates(rows)
    for k in (2, 3, 4, 5):
        p = sv.Plan(n, "c64", g, sv.run_opts(max_fuse_k=k, arith=sv.ARITH_NATIVE))
        assert p.check() == 0
        # 200 gates, each applied in float64: 200 * 2^5 roundings of 2^-53 at most
        assert np.abs(_plan_unitary_state(sv, p, n) - oracle.run(n, g)).max() < 200 * 32 * 2.0 ** -53
