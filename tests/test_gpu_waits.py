"""Waits inside the replay kernel end when nothing moves any more, not when a replay is long: with the
bound of the polls set low, replays in which one warp legitimately has nothing to do, or very much to
do, for far longer than the bound are exact all the same."""
import numpy as np
import pytest

from paper_2602_11688_b200 import workloads as W
from tests.util import check_population

pytestmark = pytest.mark.gpu

POLLS = 1 << 12          # (a poll takes 50 to 300 ns: the bound is about a millisecond without progress)


def exact_with_few_polls(w):
    from paper_2602_11688_b200 import binding as gb
    _, refs = check_population(w, scale=1.0, debug={gb.GORGO_DEBUG_POLL_LIMIT: POLLS})                  # extended build (counters)
    check_population(w, scale=1.0, debug={gb.GORGO_DEBUG_POLL_LIMIT: POLLS}, stats=False)         # plain build
    return refs


def test_caches_that_fill_late():
    """No cache comes near its capacity in the first nine tenths: the warp that lists victims idles all
    that time, and every commit after it needs one."""
    N = 60_000
    rng = np.random.default_rng(1)
    reqs = [(5.0 * k, int(rng.integers(1, 513)), int(rng.integers(0, 9)), [1_000 + k]) for k in range(N)]
    w = W.handmade([10.0], reqs, slots=4, cache_blocks=54_000, params=[(1.0, 1.0, 1.0)])
    refs = exact_with_few_polls(w)
    assert int(refs[0][4][3]) == N - 54_000           # evictions begin with request 54,000
