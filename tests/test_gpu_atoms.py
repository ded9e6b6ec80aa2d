"""GPU parity of the replay where the number of atoms per request (runs of blocks that always occur
together) is at an edge of a warp or beyond what shared memory stages: 0, 1, 31, 32, 33 and more atoms,
mixed with long prompts that are one atom each, which are evicted in part."""
import numpy as np
import pytest

from paper_2602_11688_b200 import workloads as W
from tests.util import check_population

pytestmark = pytest.mark.gpu


def trace_of_atoms(seed, sizes, n_req, B=512):
    """Requests of `sizes` single-block atoms each (random subsets of a pool, so no two blocks always
    occur together), and whole prompts of 40 to 90 blocks that come back unchanged or cut short."""
    rng = np.random.default_rng(seed)
    reqs, t, longs, nxt = [], 0.0, [], 10_000
    for k in range(n_req):
        t += float(rng.exponential(25.0))
        if rng.random() < 0.3:
            if longs and rng.random() < 0.6:
                ids = longs[int(rng.integers(len(longs)))]
                ids = ids[:int(rng.integers(1, len(ids) + 1))] if rng.random() < 0.5 else ids
            else:
                n = int(rng.integers(40, 91))
                ids = list(range(nxt, nxt + n)); nxt += n
                longs.append(ids)
        else:
            ids = [int(x) for x in rng.permutation(150)[:sizes[k % len(sizes)]]]
        n = len(ids)
        tok = 0 if n == 0 else (n - 1) * B + int(rng.integers(1, B + 1))
        reqs.append((t, tok, int(rng.integers(0, 30)), ids))
    return reqs


@pytest.mark.parametrize("R,sizes,C", [(2, (0, 1), 120), (5, (1, 7, 8, 9), 150), (16, (31, 32, 33), 130),
                                       (32, (64, 65, 2), 200), (33, (31, 0, 32, 1, 33), 140), (64, (96, 3), 110)])
def test_requests_with_atom_counts_at_the_edges(R, sizes, C):
    rng = np.random.default_rng(R)
    params = rng.normal(1.0, 0.3, size=(4, 3))
    params[0] = (0.0, 1.0, 0.0)                       # follow the cache
    params[1] = (0.0, 0.0, 1.0)                       # spread out: evictions everywhere
    w = W.handmade(rng.uniform(5, 80, size=R), trace_of_atoms(R, sizes, 300), slots=3, cache_blocks=C, params=params)
    _, refs = check_population(w, scale=1.0)
    assert sum(int(r[4][3]) for r in refs) > 0        # evictions happened
