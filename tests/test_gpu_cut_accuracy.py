"""The Builder's contraction where the two factors' large terms do not meet:
outcomes of small weight beside the other's, against the products' own sum; and
its rounding against exact integers, with digits at their ends and at random."""
import itertools
import math
from fractions import Fraction

import numpy as np
import pytest

from test_gpu_cut_steps import _terms, sv  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _reconstruct(sv, up, down, wa, cut_pos, wb, ka, kb):  # noqa: F811
    import torch
    out = torch.full((1 << (len(ka) + len(kb)),), float("nan"), dtype=torch.float64, device="cuda")
    dev = [[torch.from_numpy(r.copy()).cuda() for r in p] for p in (up, down)]
    sv.cut_reconstruct(*dev, wa, cut_pos, wb, keep_mask_a=sum(1 << q for q in ka), keep_mask_b=sum(1 << q for q in kb),
                       out=out)
    return out.cpu().numpy().reshape(1 << len(kb), 1 << len(ka))


@pytest.mark.parametrize("K,na,nb,weight", [
    (1, 7, 13, 2.0 ** -27), (1, 10, 10, 2.0 ** -40), (2, 9, 11, 2.0 ** -20), (3, 12, 8, 2.0 ** -12), (4, 7, 10, 2.0 ** -7)])
def test_rare_outcomes_of_the_cut(sv, K, na, nb, weight):  # noqa: F811
    """Every cut wire is |0> but for `weight`, without coherence, and each half's
    outcomes tell which: half of the probabilities of a cut are of that weight."""
    rng = np.random.default_rng(K + na)
    wa = na + K
    ka, kb, cut_pos = list(range(na)), list(range(nb)), list(range(na, wa))
    r = rng.exponential(size=(1 << K, 1 << na))
    r /= r.sum(axis=1, keepdims=True)
    xa, xb = np.arange(1 << na), np.arange(1 << nb)
    for y in range(1 << K):  # the outcomes of A that go with y, and (of equal size) of B
        for j in range(K):
            r[y, (xa >> j & 1) != (y >> j & 1)] = 0.0
    r += 0.125 * weight ** K * rng.exponential(size=r.shape) * 2.0 ** -na  # (but for a few)
    w = [math.prod(weight if y >> j & 1 else 1 - weight for j in range(K)) for y in range(1 << K)]
    up = np.zeros((3 ** K, 1 << K, 1 << na))
    for v, y in itertools.product(range(3 ** K), range(1 << K)):
        # the cuts measured in X or Y give both outcomes alike, whatever the wire is
        free = [j for j in range(K) if v // 3 ** j % 3]
        for z in itertools.product((0, 1), repeat=len(free)):
            s = y
            for j, b in zip(free, z):
                s = (s & ~(1 << j)) | (b << j)
            up[v, y] += 2.0 ** -len(free) * w[s] * r[s]
    up = up.reshape(3 ** K, 1 << wa)
    base = rng.exponential(size=(1 << K, 1 << nb)) * 2.0 ** -nb
    for y in range(1 << K):
        for j in range(K):
            base[y, (xb >> j & 1) != (y >> j & 1)] = 0.0
    down = np.zeros((4 ** K, 1 << nb))
    for s in range(4 ** K):  # |0>, |1>, |+>, |+i>: the last two an equal mixture here
        digits = [s // 4 ** j % 4 for j in range(K)]
        for y in itertools.product(*[(d,) if d < 2 else (0, 1) for d in digits]):
            down[s] += 2.0 ** -sum(d > 1 for d in digits) * base[sum(b << j for j, b in enumerate(y))]
    units = lambda p: np.ldexp(np.floor(np.ldexp(p.astype(np.longdouble), 112)), -112)  # distributions count 2^-112
    U, D = _terms(units(up), units(down), K, wa, cut_pos, nb, ka, kb)
    want = D.T @ U / 2 ** K
    # 2^-53 on every term and 2^-47 on every product, some roundings of float32's second parts: 2^-44 of the products
    tol = 2.0 ** -44 * (np.abs(D).T @ np.abs(U)) / 2 ** K
    got = _reconstruct(sv, up, down, wa, cut_pos, nb, ka, kb)
    assert (np.abs(got - want.astype(np.float64)) <= tol.astype(np.float64)).all()
    rare = (xb & ((1 << K) - 1)) == (1 << K) - 1
    assert 0 < want[rare].max() < 16 * weight ** K  # the small ones are there


def _exact(up, down, K, na, columns):
    """U and D as float64, from exact sums rounded once; D at the given columns only."""
    one = 1 << 112
    mu = [[int(Fraction(x) * one) for x in row] for row in up]
    U = []
    for code in itertools.product(range(4), repeat=K):
        code = code[::-1]  # code[j]: term of cut j; the list runs over the lowest cut's fastest
        v = sum((0 if t <= 1 else t - 1) * 3 ** j for j, t in enumerate(code))
        row = []
        for x in range(1 << na):
            u = 0
            for y in range(1 << K):
                f = 1
                for j, t in enumerate(code):
                    bit = y >> j & 1
                    f *= (2 if bit == t else 0) if t <= 1 else 1 - 2 * bit
                if f:
                    u += f * mu[v][x | y << na]
            row.append(float(Fraction(u, one)))
        U.append(row)
    rows = [(1, 0, 0, 0), (0, 1, 0, 0), (-1, -1, 2, 0), (-1, -1, 0, 2)]
    D = []
    for code in itertools.product(range(4), repeat=K):
        code = code[::-1]
        row = [0] * len(columns)
        for s in itertools.product(range(4), repeat=K):
            f = math.prod(rows[t][x] for t, x in zip(code, s))
            if f:
                d = down[sum(x * 4 ** j for j, x in enumerate(s))]
                row = [a + f * int(Fraction(d[c]) * one) for a, c in zip(row, columns)]
        D.append([float(Fraction(a, one)) for a in row])
    return U, D


def _check(got, U, D, K, columns):
    """Within the bound of the digits (units of both columns' scales) and the
    result's rounding, where a code is large in both columns; else 2^-44 of the products."""
    gap = 4 if K == 1 else 3
    unit = 4 ** K * 2.0 ** -58.9 + 2.0 ** -57
    scale = lambda t: [math.frexp(max(abs(r[x]) for r in t))[1] for x in range(len(t[0]))]
    ea, eb = scale(U), scale(D)
    digits = 0
    for i, c in enumerate(columns):
        for x in range(len(U[0])):
            terms = [Fraction(u[x]) * Fraction(d[i]) for u, d in zip(U, D)]
            want, size = sum(terms) / 2 ** K, sum(map(abs, terms)) / 2 ** K
            if any(abs(u[x]) >= 2.0 ** (ea[x] - gap) and abs(d[i]) >= 2.0 ** (eb[i] - gap) for u, d in zip(U, D)):
                tol = Fraction(unit) * Fraction(2) ** (ea[x] + eb[i] - K) + abs(want) / 2 ** 53
                digits += 1
            else:
                tol = size / 2 ** 44
            assert abs(Fraction(float(got[c, x])) - want) <= tol, (c, x)
    return digits


@pytest.mark.parametrize("K", [1, 2, 3])
def test_rounding_with_random_digits(sv, K):  # noqa: F811
    na, nb = 7, 13
    rng = np.random.default_rng(K)
    up = rng.exponential(size=(3 ** K, 1 << (na + K))) * 2.0 ** -na
    down = rng.exponential(size=(4 ** K, 1 << nb)) * 2.0 ** -nb
    got = _reconstruct(sv, up, down, na + K, list(range(na, na + K)), nb, list(range(na)), list(range(nb)))
    columns = [0, 31, 32, 63, (1 << nb) - 1] + rng.integers(0, 1 << nb, 11).tolist()
    assert _check(got, *_exact(up, down, K, na, columns), K, columns) > 1000


@pytest.mark.parametrize("digit", [-128, 127, 85])
@pytest.mark.parametrize("K", [1, 2, 3])
def test_rounding_with_digits_at_their_ends(sv, K, digit):  # noqa: F811
    """All terms the same number, whose digits are all the same: the products of every level add up."""
    na, nb = 7, 13
    u = 33 / 64 + sum(digit * 2.0 ** (-6 - 8 * i) for i in range(1, 6))
    up, down = np.zeros((3 ** K, 1 << K, 1 << na)), np.zeros((4 ** K, 1 << nb))
    for v, y in itertools.product(range(3 ** K), range(1 << K)):  # I/Z: 1/2, 1/2; X and Y: 1, 0
        up[v, y] = u * math.prod((0.5 if v // 3 ** j % 3 == 0 else 1 - (y >> j & 1)) for j in range(K))
    for s in range(4 ** K):  # |0> and |1>: 1; |+> and |+i>: 3/2
        down[s] = u * math.prod(1 if s // 4 ** j % 4 < 2 else 1.5 for j in range(K))
    got = _reconstruct(sv, up.reshape(3 ** K, -1), down, na + K, list(range(na, na + K)), nb, list(range(na)),
                       list(range(nb)))
    columns = [0, (1 << nb) - 1]
    U, D = _exact(up.reshape(3 ** K, -1), down, K, na, columns)
    assert all(x == u for t in (U, D) for row in t for x in row)
    _check(got, U, D, K, columns)
    assert (got == got[0, 0]).all()
