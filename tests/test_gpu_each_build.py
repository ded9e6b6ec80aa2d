"""Every build of the replay kernel on every part of the model.  Which build a launch takes depends on the number of
its candidates, and the other parity tests launch few: here the build is chosen by the test switch, for the
model parts, the waits, prompts longer than a stage, states that go on, and traces long enough for the
pipelines to settle."""
import numpy as np
import pytest

from paper_2602_11688_b200 import workloads as W
from tests import test_gpu_append as append
from tests import test_gpu_atoms as atoms
from tests import test_gpu_index as index
from tests import test_gpu_parity as parity
from tests import test_gpu_paths as paths
from tests import test_gpu_policies as policies
from tests import test_gpu_rtt as rtt
from tests import test_gpu_service as service
from tests import test_gpu_speeds as speeds
from tests import test_gpu_tuning as tuning
from tests import test_gpu_waits as waits
from tests.util import check_population, gpu_eval

pytestmark = pytest.mark.gpu

BUILDS = (1, 2, 3)


@pytest.fixture(params=BUILDS, autouse=True)
def build(request, monkeypatch):
    """Every simulator that a test creates launches this build."""
    from paper_2602_11688_b200 import binding as gb
    create = gb.gorgo_sim_create

    def create_with_build(*a, **k):
        rc, h = create(*a, **k)
        if rc == gb.GORGO_OK:
            assert gb.gorgo_debug_set(h, gb.GORGO_DEBUG_BUILD, request.param) == gb.GORGO_OK
        return rc, h
    monkeypatch.setattr(gb, "gorgo_sim_create", create_with_build)
    return request.param


CASES = [
    ("small traces, 3 replicas", parity.test_small_traces_all_mask_widths, dict(R=3, normalised=False, structured=False)),
    ("small traces, 64 replicas", parity.test_small_traces_all_mask_widths, dict(R=64, normalised=True, structured=True)),
    ("infinite and NaN scores", parity.test_huge_weights_give_infinite_and_nan_scores_like_the_scan, {}),
    ("empty, long, exact prompts", parity.test_edge_cases_empty_prompt_long_prompt_exact_fit_and_saturated_slot, {}),
    ("atom counts, 16 replicas", atoms.test_requests_with_atom_counts_at_the_edges, dict(R=16, sizes=(31, 32, 33), C=130)),
    ("atom counts, 33 replicas", atoms.test_requests_with_atom_counts_at_the_edges, dict(R=33, sizes=(31, 0, 32, 1, 33), C=140)),
    ("long prompts, 17 replicas", paths.test_prompts_longer_than_a_stage, dict(R=17, max_blocks=300, C=650)),
    ("long prompts, 64 replicas", paths.test_prompts_longer_than_a_stage, dict(R=64, max_blocks=600, C=600)),
    ("nothing ahead, 9 replicas", paths.test_small_traces_with_nothing_prepared_ahead, dict(R=9, structured=False, probe_off=1, scout_off=1)),
    ("nothing staged, 33 replicas", paths.test_small_traces_with_nothing_prepared_ahead, dict(R=33, structured=False, probe_off=1, scout_off=0)),
    ("nothing listed, 64 replicas", paths.test_small_traces_with_nothing_prepared_ahead, dict(R=64, structured=True, probe_off=0, scout_off=1)),
    ("nothing ahead, long trace", paths.test_longctx_reduced_with_nothing_prepared_ahead, dict(probe_off=1, scout_off=1)),
    ("a wait that runs out", paths.test_a_wait_that_runs_out_is_reported_and_nothing_hangs, {}),
    ("speeds, 3 replicas", speeds.test_population_with_replica_speeds, dict(R=3)),
    ("speeds, 64 replicas", speeds.test_population_with_replica_speeds, dict(R=64)),
    ("slow-down and budget, 16 replicas", service.test_population_with_the_extended_service_model, dict(R=16, slots=5, slowdown=0.15, budget=2500)),
    ("slow-down and budget, 64 replicas", service.test_population_with_the_extended_service_model, dict(R=64, slots=3, slowdown=0.15, budget=2500)),
    ("slow-down, budget, speeds", service.test_regions_reduced_with_slowdown_and_budget_and_replica_speeds, {}),
    ("service model on a state", service.test_hand_cases_and_batches_on_a_persistent_state, {}),
    ("moving network, 17 replicas", rtt.test_population_under_a_changing_network, dict(R=17, G=2)),
    ("moving network, 64 replicas", rtt.test_population_under_a_changing_network, dict(R=64, G=1)),
    ("index, 17 replicas", index.test_population_scored_with_the_index, dict(R=17, structured=False)),
    ("index, 64 replicas", index.test_population_scored_with_the_index, dict(R=64, structured=True)),
    ("everything on", index.test_regions_reduced_with_index_and_everything_else_switched_on, {}),
    ("policies", policies.test_policies_on_small_traces, dict(R=17, structured=True)),
    ("batches on a state", parity.test_route_batch_continues_a_persistent_state, {}),
    ("small batches, tiny caches", parity.test_many_small_batches_on_tiny_caches_repeatedly, dict(R=17)),
    ("small batches, 64 replicas", parity.test_many_small_batches_on_tiny_caches_repeatedly, dict(R=64)),
    ("appended batches", append.test_appended_batches_equal_the_whole_trace, dict(R=17, structured=False)),
    ("population on a grown trace", append.test_population_on_a_grown_trace_equals_the_uploaded_one, {}),
    ("online tuner", tuning.test_online_tuning_inside_one_replay_matches_oracle,
     dict(workload="regions", kw=dict(n_requests=1500, cache_blocks=500, population=4), scale=1.0, steps=40,
          start=[2.0, 1.0, 0.05], accepts=True)),
    ("waits: caches that fill late", waits.test_caches_that_fill_late, {}),
    ("waits: a long order", waits.test_first_eviction_behind_a_long_order, {}),
    ("waits: a block in every request", waits.test_victim_whose_block_occurs_in_every_request, dict(cache_blocks=2_000)),
    ("waits: a short list", waits.test_victim_whose_block_occurs_in_every_request, dict(cache_blocks=8)),
    ("waits: completions", waits.test_completions_of_all_requests_seen_by_one, {}),
    ("waits: admission", waits.test_admission_that_waits_for_hundreds_of_slots, {}),
]


@pytest.mark.parametrize("name", [c[0] for c in CASES])
def test_parity_with_each_build(name):
    _, test, kw = next(c for c in CASES if c[0] == name)
    test(**kw)


@pytest.mark.parametrize("base,n,cache,population,stats", [
    ("longctx", 12_000, 3_000, 6, False), ("regions", 8_000, 1_500, 6, False), ("sweep", 8_000, 350, 4, False),
    ("largest", 6_000, 400, 4, False), ("longctx", 8_000, 639, 4, True), ("largest", 4_000, 300, 3, True)])
def test_long_traces_with_each_build(base, n, cache, population, stats):
    w = W.make_workload(base, n_requests=n, cache_blocks=cache, population=population)
    gpu, refs = check_population(w, stats=stats)
    assert sum(int(r[4][3]) for r in refs) > 0        # evictions happened


def test_plain_and_extended_replay_agree_at_full_size():
    """The full-size comparison with the oracle asks for the counters, which the extended build keeps; the
    plain one, which a caller without counters gets, gives the same bits for every candidate."""
    w = W.make_workload("longctx")
    params = w.params[:: max(1, w.params.shape[0] // 16)]
    plain = gpu_eval(w, params, 0.5, stats=False)
    counted = gpu_eval(w, params, 0.5, stats=True)
    for key in ("route", "hit", "digest", "p95_ttft", "p95_e2e"):
        assert np.array_equal(plain[key], counted[key]), key


def test_the_build_is_the_one_asked_for(build):
    from paper_2602_11688_b200 import binding as gb
    w = W.make_workload("tiny", n_requests=300, cache_blocks=200, population=2)
    sim = gb.GorgoSim(w)
    try:
        assert gb.gorgo_debug_set(sim.h, gb.GORGO_DEBUG_BUILD, max(BUILDS) + 1) == gb.GORGO_ERR_INVALID_ARG
        rc, n, smem = gb.gorgo_replay_occupancy(sim.h)
        assert rc == gb.GORGO_OK and n >= 2 and smem > 0
    finally:
        sim.close()


@pytest.mark.parametrize("R", [8, 16, 32, 33, 64])
def test_builds_for_large_launches_leave_room_for_as_many(R, build):
    """A launch does not know what other streams run: whichever build a launch of more than a quarter of the SMs takes, an
    SM holds as many candidates as of the densest, four or (more than 32 replicas) three; of the build for few
    at least two."""
    from paper_2602_11688_b200 import binding as gb
    w = W.handmade(np.full(R, 10.0), [(5.0 * k, 600, 2, [k, k + 1]) for k in range(50)], slots=4, cache_blocks=40,
                   params=[(1.0, 1.0, 1.0)])
    sim = gb.GorgoSim(w)
    try:
        rc, n, _ = gb.gorgo_replay_occupancy(sim.h)
    finally:
        sim.close()
    assert rc == gb.GORGO_OK and n >= (2 if build == 1 else 3 if R > 32 else 4)
