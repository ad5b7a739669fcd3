"""Norms and marginals where the form for small states ends: one vector a thread or
several, one step a task or several, tasks of few and of many steps."""
import math

import numpy as np
import pytest

from test_gpu_readout import _state, sv  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n", [("c64", 15), ("c64", 16), ("c64", 17), ("c128", 15), ("c128", 16), ("c128", 17),
                                     ("c128", 18), ("c128", 19), ("c64", 19), ("c64", 20)])
def test_sums_on_both_sides_of_the_rules(sv, dtype, n):  # noqa: F811
    """Exact sums (float64 squares rounded first, 2^-53 relatively; every term
    truncated at 2^-124), rounded once."""
    a = _state(n, dtype, n, False)
    re, im = a.real.astype(np.float64), a.imag.astype(np.float64)
    parts = np.stack([re ** 2, im ** 2], axis=1)
    with sv.State(n, dtype) as s:
        s.set_amplitudes(a)
        want = math.fsum(parts.ravel())
        assert abs(s.norm() - want) <= 2.0 ** -52 * want + 2.0 ** -100
        for bits in ([0], [n - 1], [2, n - 2], [0, 3, 5, n - 3, n - 1], list(range(n - 8, n))):
            view = np.moveaxis(parts.reshape([2] * n + [2]), [n - 1 - q for q in reversed(bits)], range(len(bits)))
            view = view.reshape(1 << len(bits), -1)
            got = s.marginal_probabilities(sum(1 << q for q in bits))
            for b, row in enumerate(view):
                want = math.fsum(row)
                assert abs(got[b] - want) <= 2.0 ** -52 * want + 2.0 ** -100, (bits, b)
