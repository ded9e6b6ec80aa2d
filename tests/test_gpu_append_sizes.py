"""Growing traces where the appending launch changes form: requests just below and above what one
launch carries, and more requests in flight at the trace's end than a block has threads."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import gorgo_oracle as O
from paper_2602_11688_b200 import workloads as W
from tests.test_gpu_append import _create, _route_all


def _check(w, plan):
    ref = O.replay(w, w.params[0], 1.0)
    h = _create(w)
    try:
        from paper_2602_11688_b200 import binding as gb
        import torch
        rc, nbytes = gb.gorgo_trace_bytes(w.n_requests, int(w.hash_off[-1]))
        assert rc == gb.GORGO_OK
        buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        assert gb.gorgo_trace_begin(h, w.n_requests, int(w.hash_off[-1]), buf) == gb.GORGO_OK
        route, hit, ttft, e2e, digest = _route_all(h, w, 0, 1.0, plan)
    finally:
        gb.gorgo_sim_destroy(h)
    out = ref[0]
    assert (route == out.route).all() and (hit == out.hit).all()
    assert (ttft == out.ttft).all() and (e2e == out.e2e).all()
    assert (digest == ref[3]).all()


@pytest.mark.parametrize("blocks", [1, 107, 108, 109, 160, 161, 162, 163, 700])
def test_requests_around_one_launch(blocks):
    rng = np.random.default_rng(blocks)
    reqs, fresh = [], 0
    for k in range(12):
        shared = 0 if k == 0 else int(rng.integers(0, blocks + 1))
        ids = (reqs[-1][3][:shared] if k else []) + list(range(10_000 + fresh, 10_000 + fresh + blocks - shared))
        fresh += blocks
        reqs.append((5.0 * k, blocks * W.BLOCK_TOKENS, 4, ids))
    w = W.handmade(rng.uniform(5, 60, size=3), reqs, slots=2, cache_blocks=3 * blocks // 2 + 1,
                   params=rng.normal(1, .3, size=(1, 3)))
    _check(w, [(k + 1, k + 1) for k in range(len(reqs))])


@pytest.mark.parametrize("step", [1, 70])
def test_many_requests_in_flight_at_the_end(step):
    rng = np.random.default_rng(step)
    reqs = [(2.0 * k, W.BLOCK_TOKENS, int(rng.integers(1, 60)), [int(rng.integers(0, 40))]) for k in range(450)]
    w = W.handmade(rng.uniform(5, 60, size=5), reqs, slots=8, cache_blocks=9, params=rng.normal(1, .3, size=(1, 3)))
    _check(w, [(k, k) for k in range(step, 450, step)] + [(450, 450)])
