"""GPU parity at the edges of the rule that picks the replay kernel's build: up to a quarter of the SMs, up to
two candidates an SM, more.  Traces that make the rare paths of the eviction common: a prompt that many share, caches of a few
prompts, victims that occur again between their listing and their eviction."""
import numpy as np
import pytest

from paper_2602_11688_b200 import workloads as W
from tests.util import assert_candidate_matches, gpu_eval, oracle_eval, small_trace

pytestmark = pytest.mark.gpu


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def shared_prompt_trace(seed, n_req, B=512):
    """Sessions that all begin with one of two prompts of two blocks."""
    reqs = []
    for t, in_tok, out, ids in small_trace(seed, n_req=n_req, n_sessions=20, max_blocks=9):
        reqs.append((t, in_tok + 2 * B, out, ([1, 2] if ids[0] % 3 else [3, 4]) + list(ids)))
    return reqs


@pytest.mark.parametrize("per_sm,extra", [(0, 3), (1, 0), (1, 1), (2, 0), (2, 1), (4, 5)])
@pytest.mark.parametrize("R,C,stats", [(2, 24, False), (8, 17, True), (32, 40, False), (33, 13, True), (64, 30, False)])
def test_every_build_matches_the_oracle(per_sm, extra, R, C, stats):
    rng = np.random.default_rng(R)
    base = rng.normal(1.0, 0.3, size=(3, 3))
    base[0] = (0.0, 1.0, 0.0)                         # follow the cache
    base[1] = (0.0, 0.0, 1.0)                         # spread out: evictions everywhere
    w = W.handmade(rng.uniform(5, 60, size=R), shared_prompt_trace(R, 400), slots=2, cache_blocks=C, params=base)
    P = per_sm * _sms() + extra
    params = np.tile(base, (P // 3 + 1, 1))[:P]
    gpu = gpu_eval(w, params, 1.0, stats=stats)
    refs = oracle_eval(w, base, 1.0)
    for p in sorted({0, 1, 2, P - 3, P - 2, P - 1}):
        assert_candidate_matches(gpu, p, refs[p % 3])
    for key in ("route", "hit", "p95_ttft", "p95_e2e"):   # equal weights, equal results
        for k in range(3):
            assert (gpu[key][k::3] == gpu[key][k]).all(), (key, k)
    assert sum(int(r[4][3]) for r in refs) > 0        # evictions happened


@pytest.mark.parametrize("over", [0, 1])
@pytest.mark.parametrize("R,C,stats", [(8, 17, True), (32, 40, False), (64, 30, False)])
def test_the_last_population_of_the_build_for_few_and_the_next(over, R, C, stats):
    test_every_build_matches_the_oracle(0, _sms() // 4 + over, R, C, stats)


@pytest.mark.parametrize("lam,steps,resident", [(1, 2, 1), (5, 3, 1), (5, 3, 5), (5, 3, 6), (4, 0, 4)])
def test_the_parent_is_evaluated_with_the_first_offspring(lam, steps, resident):
    """Workspaces that hold the first population and the parent, the population alone, or one candidate."""
    from oracle import gorgo_oracle as O
    from oracle import gorgo_tuning as T
    from paper_2602_11688_b200 import binding as gb
    rng = np.random.default_rng(lam)
    w = W.handmade(rng.uniform(5, 60, size=4), small_trace(3, n_req=300), slots=2, cache_blocks=15,
                   params=[(0.5, 1.0, 0.1)])
    z = rng.standard_normal((steps, lam, 2))
    es = dict(tuned=np.array([0, 2], np.uint32), lo=np.array([0.05, 0.05]), hi=np.array([2.0, 0.5]))
    sim = gb.GorgoSim(w)
    try:
        sim.ensure_workspace(resident)
        rc, x, f, sigma, hist = gb.gorgo_es_run(sim.h, x0=w.params[0], z=z, sigma0=0.5, sigma_up=1.5, n_steps=steps, lam=lam,
                                                workspace=sim.workspace, stream=sim.stream, time_scale=1.0, **es)
        assert rc == gb.GORGO_OK
    finally:
        sim.close()
    rx, rf, rsigma, rhist = T.es_run(lambda v: O.replay(w, np.array(v), 1.0)[1], w.params[0].tolist(), es["tuned"].tolist(),
                                     es["lo"].tolist(), es["hi"].tolist(), 0.5, 1.5, z.tolist())
    assert x.tolist() == rx and f == rf and sigma == rsigma
    for t, h in enumerate(rhist):
        assert hist[t, 0] == h[0] and bool(hist[t, 1]) == h[1] and hist[t, 3] == h[3], t


@pytest.mark.parametrize("steps,lam", [(0, 3), (1, 1), (2, 3)])
@pytest.mark.parametrize("R", [4, 40])
def test_the_strategy_asks_for_the_workspace_of_one_candidate(R, steps, lam):
    """The same with and without steps; one byte less is refused and nothing is written."""
    import torch
    from paper_2602_11688_b200 import binding as gb
    w = W.handmade(np.linspace(5.0, 60.0, R), small_trace(3, n_req=200), slots=2, cache_blocks=15, params=[(0.5, 1.0, 0.1)])
    z = np.random.default_rng(1).standard_normal((steps, lam, 2))
    sim = gb.GorgoSim(w)
    try:
        rc, need = gb.gorgo_workspace_bytes(sim.h, 1)
        room = torch.zeros(need, dtype=torch.uint8, device="cuda")
        kw = dict(x0=w.params[0], z=z, tuned=[0, 2], lo=[0.05, 0.05], hi=[2.0, 0.5], sigma0=0.5, sigma_up=1.5, n_steps=steps,
                  lam=lam, stream=sim.stream, time_scale=1.0)
        assert gb.gorgo_es_run(sim.h, workspace=room[:need - 1], **kw)[0] == gb.GORGO_ERR_WORKSPACE_TOO_SMALL
        torch.cuda.synchronize()
        assert int(room.count_nonzero()) == 0
        assert gb.gorgo_es_run(sim.h, workspace=room, **{**kw, "time_scale": -1.0})[0] == gb.GORGO_ERR_NONFINITE_PARAM
        assert gb.gorgo_es_run(sim.h, workspace=room, **kw)[0] == gb.GORGO_OK
    finally:
        sim.close()


@pytest.mark.parametrize("R,C", [(8, 17), (40, 30)])
def test_populations_on_several_streams_at_once(R, C):
    """Launches of all builds side by side, on streams of their own, give what each gives alone."""
    import torch
    from paper_2602_11688_b200 import binding as gb
    base = np.random.default_rng(R).normal(1.0, 0.3, size=(8, 3))
    w = W.handmade(np.linspace(5.0, 60.0, R), shared_prompt_trace(R, 600), slots=2, cache_blocks=C, params=base)
    sizes = [_sms() // 4, _sms(), _sms() + 1, 2 * _sms() + 3]
    sims = [gb.GorgoSim(w) for _ in sizes]
    try:
        params = [np.tile(base, (P // 8 + 1, 1))[:P] for P in sizes]
        alone = [gpu_eval(w, p, 1.0, stats=False, sim=s) for s, p in zip(sims, params)]
        refs = oracle_eval(w, base[:2], 1.0)
        for got in alone:
            for p in (0, 1):
                assert_candidate_matches(got, p, refs[p])
        streams = [torch.cuda.Stream() for _ in sizes]
        for _ in range(3):
            outs = []
            torch.cuda.synchronize()
            for sim, p, st in zip(sims, params, streams):
                with torch.cuda.stream(st):
                    outs.append(sim.eval_population(p, 1.0, want_route=True, want_hit=True, want_digest=True))
            torch.cuda.synchronize()
            for got, want in zip(outs, alone):
                for key in ("status", "route", "hit", "digest", "p95_ttft", "p95_e2e"):
                    assert np.array_equal(got[key].cpu().numpy(), want[key]), key
    finally:
        for sim in sims:
            sim.close()


def test_the_occupancy_reported_is_of_the_build_that_a_launch_takes():
    from paper_2602_11688_b200 import binding as gb
    w = W.handmade(np.linspace(5.0, 60.0, 16), small_trace(3, n_req=100), slots=2, cache_blocks=15, params=[(0.5, 1.0, 0.1)])
    sim = gb.GorgoSim(w)
    try:
        by_build = {}
        for build in (1, 2, 3):
            assert gb.gorgo_debug_set(sim.h, gb.GORGO_DEBUG_BUILD, build) == gb.GORGO_OK
            by_build[build] = gb.gorgo_replay_occupancy(sim.h)
        sms = _sms()
        for candidates, build in ((1, 1), (sms // 4, 1), (sms // 4 + 1, 2), (2 * sms, 2), (2 * sms + 1, 3)):
            assert sim.replay_occupancy(candidates) == by_build[build], candidates
        assert gb.gorgo_replay_occupancy(sim.h) == by_build[3]
    finally:
        sim.close()
