"""The tile pass of few tiles (two copies of the tile in shared memory, shared by
a cluster where SMs would be idle) against the general one: both form every sum in the same order, so a state run by
itself (few tiles) and the same state among enough others (more tiles than SMs)
have the same bits, over tile sizes, odd state sizes, every gate and block width."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import _random_circuit

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


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("dtype,n,tile", [
    ("c64", 1, 0), ("c64", 7, 0), ("c64", 13, 0), ("c64", 18, 13), ("c64", 21, 13), ("c64", 11, 11), ("c64", 14, 10), ("c64", 15, 12), ("c64", 16, 13),
    ("c128", 2, 0), ("c128", 8, 0), ("c128", 10, 0), ("c128", 12, 0), ("c128", 17, 12), ("c128", 13, 9), ("c128", 14, 11), ("c128", 16, 12)])
def test_same_bits_as_the_general_pass(sv, dtype, n, tile, k):
    arith = sv.ARITH_NATIVE if dtype == "c64" else sv.ARITH_DF64
    opts = sv.run_opts(arith=arith, max_fuse_k=k, tile_qubits=tile)
    g = _random_circuit(n, 90 if n > 1 else 20, 50 * n + k)  # more than 48 ops in a pass when k = 1
    copies = max(1, 600 >> max(0, n - (tile or 13)))
    with sv.Batch([(n, dtype, g, None)] * copies, opts) as b:
        many = b.execute()
    with sv.State(n, dtype) as s:
        s.apply_circuit(g, opts)
        assert s.stats()["arith"] == arith
        p = s.probabilities()
    for q in many:
        assert np.array_equal(p, q)
    # 90 gates of at most 32 terms each, 90 * 32 ulps of 1 (2^-24, 2^-48), in squares twice that
    tol = 2 * 90 * 32 * 2.0 ** (-24 if dtype == "c64" else -48)
    assert np.abs(p - oracle.probabilities(oracle.run(n, g))).max() <= tol
