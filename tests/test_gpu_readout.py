"""Read-out kernels on the GPU: probabilities rounded once, marginals and norms
summed exactly, over widths, masks and magnitudes at the edges of their paths."""
import math
from fractions import Fraction

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


def _state(n, dtype, seed, wide):
    """Random amplitudes of norm at most 1; wide: magnitudes over the whole range of the type, zeros and subnormals."""
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((1 << n, 2)) / 2 ** (n / 2 + 1)
    if wide:
        a *= 2.0 ** rng.integers(-140 if dtype == "c64" else -500, 1, size=a.shape)
        a[rng.random(a.shape) < 0.2] = 0.0
    return np.ascontiguousarray(a).view(np.complex128)[:, 0].astype(np.complex64 if dtype == "c64" else np.complex128)


def _probs(a):
    """|a|^2 rounded once: float32 squares are exact in float64, so numpy's sum is; float64 from exact fractions."""
    if a.dtype == np.complex64:
        return a.real.astype(np.float64) ** 2 + a.imag.astype(np.float64) ** 2
    return np.array([float(Fraction(float(z.real)) ** 2 + Fraction(float(z.imag) * float(z.imag))) for z in a])


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("n", [1, 2, 3, 12])
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_probabilities_are_rounded_once(sv, dtype, n, wide):
    import torch
    a = _state(n, dtype, 17 * n + wide, wide)
    with sv.State(n, dtype) as s:
        s.set_amplitudes(a)
        assert np.array_equal(s.probabilities(), _probs(a))
        odd = torch.empty((1 << n) + 1, dtype=torch.float64, device="cuda")[1:]  # 8-byte aligned only
        assert np.array_equal(s.probabilities(odd).cpu().numpy(), _probs(a))


@pytest.mark.parametrize("n", [1, 2, 5, 6, 7, 11, 14])
@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_marginals_and_norm_are_exact_sums(sv, dtype, n):
    """Each bin is the exact sum of its probabilities (float64 ones rounded
    first, a relative error of at most 2^-53; every term truncated at 2^-124),
    rounded once: within 2^-52 relatively, plus 2^-100."""
    a = _state(n, dtype, 5 * n, False)
    rng = np.random.default_rng(n)
    masks = {0, (1 << n) - 1, 1, 1 << (n - 1)} | {int(rng.integers(1 << n)) for _ in range(6)}
    idx = np.arange(1 << n)
    re, im = a.real.astype(np.float64), a.imag.astype(np.float64)
    with sv.State(n, dtype) as s:
        s.set_amplitudes(a)
        for mask in masks:
            bits = [q for q in range(n) if mask >> q & 1]
            bin_of = sum(((idx >> q) & 1) << j for j, q in enumerate(bits)) if bits else np.zeros_like(idx)
            got = s.marginal_probabilities(mask)
            for b in range(len(got)):
                pick = bin_of == b
                want = math.fsum(np.concatenate([re[pick] ** 2, im[pick] ** 2]))
                assert abs(got[b] - want) <= 2.0 ** -52 * want + 2.0 ** -100, (mask, b)
        want = math.fsum(np.concatenate([re ** 2, im ** 2]))
        assert abs(s.norm() - want) <= 2.0 ** -52 * want + 2.0 ** -100
