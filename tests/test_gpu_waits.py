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


LONG = 60_000            # requests behind one step of another warp


def fleet_of_two(reqs, cache_blocks):
    """Requests (replica, output tokens, block ids): the network term alone decides, by the origin."""
    t = [(2.0 * k, 512 * len(ids), out, ids) for k, (_, out, ids) in enumerate(reqs)]
    return W.handmade([[10.0, 90.0], [90.0, 10.0]], t, slots=4, cache_blocks=cache_blocks, n_regions=2,
                      origin=[x[0] for x in reqs], params=[(1.0, 0.0, 0.0)])


def test_first_eviction_behind_a_long_order():
    """The cache is far from full until one prompt needs all of it: the whole order of the replica, most
    of it superseded, is walked while that one commit waits."""
    reqs = [(2.0 * k, 512, 1, [1]) for k in range(LONG)]
    reqs += [(2.0 * (LONG + k), 512 * 2_000, 1, list(range(10_000 * (k + 1), 10_000 * (k + 1) + 2_000))) for k in range(3)]
    w = W.handmade([10.0], reqs, slots=4, cache_blocks=2_000, params=[(1.0, 1.0, 1.0)])
    assert int(exact_with_few_polls(w)[0][4][3]) == 1 + 2 * 2_000


@pytest.mark.parametrize("cache_blocks", [2_000, 8])
def test_victim_whose_block_occurs_in_every_request(cache_blocks):
    """Replica 1 sees a block once, replica 0 after that in every request; then replica 1 has to evict it.
    2,000 blocks: nothing is listed ahead and the scout walks all occurrences; 8: the block is listed at
    once and the commit walks what occurred since."""
    reqs = [(1, 1, [7])] + [(0, 1, [7])] * LONG
    reqs += [(1, 1, list(range(10_000 * (k + 1), 10_000 * (k + 1) + cache_blocks))) for k in range(3)]
    refs = exact_with_few_polls(fleet_of_two(reqs, cache_blocks))
    assert int(refs[0][4][3]) == 1 + 2 * cache_blocks


def test_replica_with_few_requests_in_a_long_log():
    """Nearly all requests go to replica 0; the order of replica 1 lies thousands of log words apart."""
    reqs = [((1 if k % 20_000 == 5 else 0), 1, [1 + k % 3]) for k in range(4 * LONG)]
    reqs += [(1, 1, list(range(10_000 * (k + 1), 10_000 * (k + 1) + 2_000))) for k in range(3)]
    exact_with_few_polls(fleet_of_two(reqs, 2_000))


def test_completions_of_all_requests_seen_by_one():
    """All requests are in flight at once and done before the next arrival: their completions are one
    list of that request."""
    reqs = [(0.001 * k, 512, 1, [k % 5]) for k in range(LONG)]
    reqs += [(1e9 + 100.0 * k, 512, 3, [k % 7]) for k in range(300)]
    w = W.handmade([10.0, 11.0, 12.0], reqs, slots=16, cache_blocks=4, params=[(1.0, 1.0, 1.0)])
    exact_with_few_polls(w)


def test_admission_that_waits_for_hundreds_of_slots():
    """A KV budget of one request and thousands of slots: every request moves past the finish of all before
    it, and each of these rounds looks at all slots."""
    from paper_2602_11688_b200 import binding as gb
    from oracle import gorgo_oracle as O
    import torch
    N = 300
    reqs = [(0.01 * k, 512, 3, [k]) for k in range(N)]
    w = W.handmade([10.0], reqs, slots=2_048, cache_blocks=64, params=[(1.0, 1.0, 1.0)])
    sim = gb.GorgoSim(w)
    assert gb.gorgo_sim_set_service_model(sim.h, 0.0, 515) == gb.GORGO_OK
    assert gb.gorgo_debug_set(sim.h, gb.GORGO_DEBUG_POLL_LIMIT, POLLS) == gb.GORGO_OK
    out = sim.eval_population(w.params, 1.0, want_route=True)
    torch.cuda.synchronize()
    assert int(out["status"].item()) == 0
    _, p95_ttft, p95_e2e, _, _ = O.replay(w, w.params[0], 1.0, kv_budget_tokens=515)
    assert float(out["p95_ttft"].item()) == p95_ttft and float(out["p95_e2e"].item()) == p95_e2e
    sim.close()
