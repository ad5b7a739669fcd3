"""Probabilities of a batch: states of fewer, as many and more amplitudes than a
block of the launch, in any order, more blocks than CTAs, outputs of 8-byte alignment;
and passes of states of every width in one launch of either kernel."""
import numpy as np
import pytest

from test_gpu_parity import _random_circuit
from test_gpu_readout import sv  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [0, 1, 4])  # one-qubit blocks take the general pass in a batch, wide ones the few-tile pass
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_every_state_has_its_own(sv, dtype, k):  # noqa: F811
    import torch
    widths = [1, 14, 10, 11, 12, 2, 13, 5] + [3] * 1300 + [12, 1, 11]
    circuits = {n: _random_circuit(n, 20, 7 * n) for n in set(widths)}
    buffers = [torch.full(((1 << n) + 1,), float("nan"), dtype=torch.float64, device="cuda") for n in widths]
    opts = sv.run_opts(arith=sv.ARITH_NATIVE if dtype == "c64" else sv.ARITH_DF64, max_fuse_k=k)
    with sv.Batch([(n, dtype, circuits[n], b[i % 2:][: 1 << n]) for i, (n, b) in enumerate(zip(widths, buffers))], opts) as b:
        b.execute()
    want = {}
    for n, g in circuits.items():
        with sv.State(n, dtype) as s:
            s.apply_circuit(g, opts)
            want[n] = s.probabilities()
    for i, (n, b) in enumerate(zip(widths, buffers)):
        got = b.cpu().numpy()
        assert np.array_equal(got[i % 2:][: 1 << n], want[n]), i
        assert np.isnan(got[0] if i % 2 else got[-1])  # and nothing beside them
