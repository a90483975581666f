"""The warp's box search on the CPU: a replay of its steps (32 starts compared
at a time) against the bisection, for every number of boxes and with empty
boxes, whose starts repeat."""
import numpy as np
import pytest


def _warp_search(starts, i):
    lo, n = 0, len(starts)
    while n > 1:
        step = (n + 31) >> 5
        below = [lane * step < n and starts[lo + lane * step] <= i for lane in range(32)]
        k = max(sum(below) - 1, 0)
        lo += k * step
        n = min(step, n - k * step)
    return lo


@pytest.mark.parametrize("nbox", [1, 2, 31, 32, 33, 63, 64, 65, 512, 1023, 1024, 1025, 1056, 1057, 40_000])
@pytest.mark.parametrize("empty", [0.0, 0.5, 0.95])
def test_warp_search_equals_bisection(nbox, empty):
    rng = np.random.default_rng(nbox)
    ns = rng.integers(1, 50, nbox) * (rng.random(nbox) >= empty)
    starts = np.concatenate([[0], np.cumsum(ns)[:-1]])
    total = int(ns.sum())
    for i in {0, max(total - 1, 0), total, *map(int, starts[rng.integers(0, nbox, 40)]),
              *map(int, rng.integers(0, total + 1, 60))}:
        assert _warp_search(starts, i) == np.searchsorted(starts, i, side="right") - 1
