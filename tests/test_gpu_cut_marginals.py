"""Marginals of the variants one thread a bin against warp sweeps: the same exact
sums on both sides of the rule that chooses (4 or 8 rows, bins for the chip's
threads or fewer), low and high qubits summed, odd widths, and four cuts."""
import pytest

from test_gpu_cut_steps import sv, test_reconstruct_steps as check  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _without(width, *summed):
    return [q for q in range(width) if q not in summed]


@pytest.mark.parametrize("K,wa,wb,ka,kb", [
    (1, 16, 3, _without(15, 6, 9), [1]),           # 4 rows, 3 * 2^14 bins
    (1, 16, 3, _without(15, 6, 9, 0), [0, 2]),     # 4 rows, 3 * 2^13
    (1, 16, 5, _without(15, 7, 10, 13), [3]),      # 8 rows
    (1, 15, 8, _without(14, 0, 5), [7]),           # no row
    (1, 15, 6, _without(14), [0, 1, 2, 3, 4, 5]),  # nothing summed
    (1, 2, 16, [], _without(16, 1, 2, 11, 15)),    # 4 rows downstream, the highest summed
    (2, 14, 12, _without(12, 2), _without(12, 3, 8)), (4, 9, 9, _without(5, 4), _without(9, 0, 8))])
def test_bins_and_sweeps(sv, K, wa, wb, ka, kb):  # noqa: F811
    check(sv, K, wa, wb, ka, kb)
