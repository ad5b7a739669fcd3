"""complex64 norms and marginals at the edges of the two-integer split of a
component (its window depends on the width): the exact sums, rounded once."""
import math

import numpy as np
import pytest

from test_gpu_readout import sv  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4, 9, 13, 18])
def test_sums_at_the_window_edges(sv, n):  # noqa: F811
    h = (n + 1) // 2 - 4
    rng = np.random.default_rng(n)
    size = 2 << n
    # full mantissas just inside and outside 2^-h, around the lowest bit 2^(-h - 43), below it, subnormals, zeros
    exps = rng.choice([-h, -h - 1, -h - 5, -h - 19, -h - 20, -h - 21, -h - 30, -h - 42, -h - 43, -h - 44, -130, -149], size)
    v = np.ldexp(1 + rng.integers(0, 1 << 23, size) / 2.0 ** 23, exps).astype(np.float32)
    exact = np.ldexp(1.0, np.array([-h, -h - 1, -h - 21, -h - 43])).astype(np.float32)
    v[: min(size, 4)] = exact[: min(size, 4)]
    big = np.flatnonzero(v > 2.0 ** (-h - 3))
    v[big[8:]] = 0.0  # (a norm of the order of one)
    v[rng.random(size) < 0.1] = 0.0
    v *= rng.choice([-1, 1], size).astype(np.float32)
    v *= np.float32(0.125) if h < 1 else np.float32(1)
    a = v.reshape(-1, 2).copy().view(np.complex64)[:, 0]
    re, im = a.real.astype(np.float64), a.imag.astype(np.float64)
    idx = np.arange(1 << n)
    with sv.State(n, "c64") as s:
        s.set_amplitudes(a)
        want = math.fsum(np.concatenate([re ** 2, im ** 2]))
        # each term truncated at 2^-124 and the sum rounded once
        assert abs(s.norm() - want) <= 2.0 ** -52 * want + size * 2.0 ** -124
        for mask in {0, 1, (1 << n) - 1, int(rng.integers(1 << n)) & 0x3ff}:
            bits = [q for q in range(n) if mask >> q & 1]
            if len(bits) > 8 and n > 9:
                continue
            bin_of = sum((((idx >> q) & 1) << j for j, q in enumerate(bits)), np.zeros_like(idx))
            got = s.marginal_probabilities(mask)
            for b in range(len(got)):
                pick = bin_of == b
                want = math.fsum(np.concatenate([re[pick] ** 2, im[pick] ** 2]))
                assert abs(got[b] - want) <= 2.0 ** -52 * want + size * 2.0 ** -124, (mask, b)


@pytest.mark.parametrize("apart", range(10))
def test_probabilities_by_exponent_distance(sv, apart):  # noqa: F811
    """Both squares and their sum rounded once, for components 2^apart apart,
    mantissas at their ends, the lowest normal exponents and subnormals."""
    n = 10
    rng = np.random.default_rng(apart)
    m = rng.integers(0, 1 << 23, (1 << n, 2))
    m[:: 3] = rng.choice([0, 1, (1 << 23) - 1], m[:: 3].shape)
    e = rng.integers(-100, -4, 1 << n)
    e[: 8] = [-126, -125, -119, -118, -117, -127, -140, -149]
    v = np.ldexp(1 + m / 2.0 ** 23, np.stack([e, e - apart], axis=1)).astype(np.float32)
    v[1:: 2] = v[1:: 2, ::-1]
    a = np.ascontiguousarray(v).view(np.complex64)[:, 0]
    with sv.State(n, "c64") as s:
        s.set_amplitudes(a)
        # float32 squares are exact in float64, so its sum is rounded once
        assert np.array_equal(s.probabilities(), a.real.astype(np.float64) ** 2 + a.imag.astype(np.float64) ** 2)
