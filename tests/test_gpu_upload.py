"""New traces on a kept handle: inputs that are staged on the host and copied at
once, and inputs past the stage's size, whose per-call arrays are copied from the
caller's; with and without tenants, and after a rejected upload."""
import numpy as np
import pytest

import oracle
from paper_2505_05286_gb300 import build as B
from paper_2505_05286_gb300 import hxsim as H
from paper_2505_05286_gb300 import workloads as W

FIELDS = ["p95_us", "makespan_us", "events", "digest", "slo_met", "n_done", "status"]


def _traces(recipe, n, nq, seed):
    # no corrections: every seed gives the same shapes
    r = W.Recipe(**{**recipe.__dict__, "p_err": 0.0})
    return [W.make_trace(r, 1, seed * 100 + t, n_queries=nq) for t in range(n)], W.make_cluster(r)


@pytest.mark.gpu
@pytest.mark.parametrize("tenants", [False, True])
@pytest.mark.parametrize("n,nq", [(3, 50), (38, 20000)])  # 13 KB, and 68 MB of calls (the stage holds 64)
def test_upload_replaces_every_input(n, nq, tenants):
    B.build()
    recipe = W.EXTRA["two-tenant"] if tenants else W.RECIPES[1]
    a, cl = _traces(recipe, n, nq, 1)
    b, _ = _traces(recipe, n, nq, 2)
    grid = W.subset_grid(W.make_grid(recipe), [0, 40])
    sims = [1, 2 * n - 2]  # first and last trace
    sim = H.Sim(a, cl, grid, subset=sims)
    bad = list(b)
    bad[-1] = W.Trace(**{**b[-1].__dict__, "prompt": b[-1].prompt * 0})
    for step, traces in enumerate((a, b, b, a)):
        if step == 2:  # refused: the handle keeps what it has
            with pytest.raises(H.HxError):
                sim.upload(bad)
        elif step:
            sim.upload(traces)
        sim.run()
        got = sim.results()[sims]
        want, extra = oracle.run(W.Workload("upload", traces, cl, grid, 0), sims, extra=True)
        for f in FIELDS:
            assert np.array_equal(got[f], want[f]), f
        if tenants:
            assert np.array_equal(sim.extras()[sims]["p95_us"], extra["p95_us"])
    sim.close()


@pytest.mark.gpu
@pytest.mark.parametrize("force_generic", [False, True])
@pytest.mark.parametrize("record", [(), (1,)])
def test_captured_run_follows_uploads(force_generic, record):
    """A captured run serves whatever traces are uploaded before a replay, also ones
    whose calls need 64-bit times where those at the capture did not, and back."""
    import torch
    B.build()
    recipe = W.RECIPES[1]
    a, cl = _traces(recipe, 2, 60, 1)
    b, _ = _traces(recipe, 2, 60, 2)
    b[1].prompt[::3] = 1_000_000  # past 2^25 us on the slower types
    grid = W.subset_grid(W.make_grid(recipe), [0, 40, 63])
    for first, second in ((a, b), (b, a)):
        sim = H.Sim(first, cl, grid, record_sims=record, force_generic=force_generic)
        sim.run()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            sim.run(torch.cuda.current_stream())
        for traces in (first, second, first):
            sim.upload(traces)
            graph.replay()
            torch.cuda.synchronize()
            got, wl = sim.results(), W.Workload("captured", traces, cl, grid, 0)
            want = oracle.run(wl)
            for f in FIELDS:
                assert np.array_equal(got[f], want[f]), f
            for j, s in enumerate(record):
                _, log = oracle.simulate(traces[s // 3], cl, oracle.point_of(grid, s % 3), log=True)
                for f in ("budget", "start", "end"):
                    assert np.array_equal(sim.records(j)[f], log[f]), f
        sim.close()
