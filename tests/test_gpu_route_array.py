"""The caller's route array is written and nothing else: any alignment, sizes that are no multiple of
four bytes, bytes on either side untouched and without influence, whatever they are."""
import numpy as np
import pytest

from oracle import gorgo_oracle as O
from paper_2602_11688_b200 import workloads as W
from tests.util import small_trace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 3, 5, 130, 131])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("P", [1, 3])
def test_route_array_of_any_alignment_and_size(N, shift, P):
    import torch
    from paper_2602_11688_b200 import binding as gb
    rng = np.random.default_rng(N)
    w = W.handmade(rng.uniform(5, 60, size=3), small_trace(N, n_req=N, structured=False), slots=2, cache_blocks=9,
                   params=rng.normal(1.0, 0.3, size=(P, 3)))
    refs = [O.replay(w, row, 1.0)[0].route for row in w.params]
    sim = gb.GorgoSim(w)
    sim.ensure_workspace(P)
    out = torch.empty((2, P), dtype=torch.float64, device="cuda")
    for guard in (0, 1, 2, 255):                       # (the numbers of the replicas, and none)
        buf = torch.full((8 + P * N + 8,), guard, dtype=torch.uint8, device="cuda")
        rc = gb.gorgo_eval_population(sim.h, P, w.params, 1.0, sim.workspace, sim.stream, out[0], out[1],
                                      buf[4 + shift:])
        assert rc == gb.GORGO_OK
        got = buf.cpu().numpy()
        end = 4 + shift + P * N
        assert (got[4 + shift:end].reshape(P, N) == np.stack(refs)).all()
        assert (got[:4 + shift] == guard).all() and (got[end:] == guard).all()
    sim.close()


def test_online_tuners_write_the_callers_routes():
    """Hops that are no multiple of four requests, several tuners, an array of odd alignment."""
    import torch
    from paper_2602_11688_b200 import binding as gb
    w = W.make_workload("tiny", n_requests=403, cache_blocks=150, population=3)
    sim = gb.GorgoSim(w)
    sim.ensure_workspace(3)
    rng = np.random.default_rng(0)
    kw = dict(x0=np.tile([0.5, 1.0, 0.1], (3, 1)), z=rng.standard_normal((3, 20, 2)), workspace=sim.workspace,
              stream=sim.stream, time_scale=1.0, tuned=[0, 2], lo=[0.05, 0.05], hi=[2.0, 0.5], sigma0=0.5, sigma_up=1.5,
              window=31, hop=7)
    a, b = (torch.full((3 * 403 + 16,), 9, dtype=torch.uint8, device="cuda") for _ in range(2))
    assert gb.gorgo_tune_online(sim.h, route=a, **kw)[0] == gb.GORGO_OK
    assert gb.gorgo_tune_online(sim.h, route=b[3:], **kw)[0] == gb.GORGO_OK
    assert torch.equal(a[:3 * 403], b[3:3 + 3 * 403]) and bool((a[:3 * 403] < 4).all())
    assert bool((a[3 * 403:] == 9).all()) and bool((b[:3] == 9).all()) and bool((b[3 + 3 * 403:] == 9).all())
    sim.close()
