"""The local queues and the per-call log on the GPU against the oracle: heap
sizes at the edges of its levels and regions, eight requests joining a queue at
once, equal keys, and the logged budgets of every kernel family."""
import numpy as np
import pytest

import oracle
from paper_2505_05286_gb300 import build as B
from paper_2505_05286_gb300 import hxsim as H
from paper_2505_05286_gb300 import workloads as W

FIELDS = ["p95_us", "makespan_us", "events", "digest", "slo_met", "n_done", "status"]


def _grid(policies):
    n = 2 * len(policies)
    return W.Grid(np.array([W.SCALE, W.SCALE // 2] * len(policies), np.int64),
                  np.array([W.SCALE, 4 * W.SCALE] * len(policies), np.int64), np.full(n, 2, np.int32),
                  np.full(n, 300_000 ** 2, np.int64), np.repeat(np.array(policies, np.uint8), 2),
                  np.zeros(n, np.uint8))


def _run(tr, cl, grid, record=()):
    B.build()
    wl = W.Workload("queue", [tr], cl, grid, W.OBJ_P95)
    sim = H.Sim(wl.traces, cl, grid, record_sims=record)
    sim.run()
    got, want = sim.results(), oracle.run(wl)
    for f in FIELDS:
        assert np.array_equal(got[f], want[f]), f
    for j, s in enumerate(record):
        _, lo = oracle.simulate(tr, cl, oracle.point_of(grid, s), log=True)
        lg = sim.records(j)
        for f in ("inst", "enq", "budget", "start", "end"):
            assert np.array_equal(lg[f], lo[f]), (s, f)
    family = sim.info()["generic_kernel"]
    sim.close()
    return family


def _burst(n, equal, seed):
    """n single-shot requests at time 0, then k = 8 queries while they wait."""
    rng = np.random.default_rng(seed)
    nq, k = n + 6, 8
    ks = np.zeros(nq, np.uint8)
    ks[n:] = k
    cnt = np.where(ks == 0, 1, 2 + k)
    base = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int32)
    nc = int(base[-1])
    stage, cand = np.full(nc, W.STAGE_E, np.uint8), np.zeros(nc, np.uint8)
    for i in range(n, nq):
        stage[base[i]] = W.STAGE_S
        stage[base[i] + 1:base[i] + 1 + k] = W.STAGE_G
        cand[base[i] + 1:base[i] + 1 + k] = np.arange(k)
    prompt = np.full(nc, 1000, np.int32) if equal else rng.integers(200, 6000, nc).astype(np.int32)
    arrival = np.concatenate([np.zeros(n, np.int64), 50_000 * (1 + np.arange(6, dtype=np.int64))])
    return W.Trace(arrival, ks, base, prompt, np.full(nc, 50, np.int32), np.full(nc, 50, np.int32), stage, cand,
                   np.zeros(nc, np.uint8))


@pytest.mark.gpu
@pytest.mark.parametrize("generic", [False, True])
@pytest.mark.parametrize("equal", [False, True])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 34, 1056, 1057, 1058])
@pytest.mark.parametrize("n_inst,slots", [(1, 1), (2, 16), (33, 1)])
def test_queue_sizes(n_inst, slots, n, equal, generic):
    cl = W.make_cluster(W.RECIPES[1])
    cl.inst_type = np.zeros(n_inst, np.uint8)
    cl.slots = np.array([slots] * 3, np.int32)
    _run(_burst(n, equal, n), cl, _grid([0, 1, 2] if generic else [0]))


@pytest.mark.gpu
@pytest.mark.parametrize("equal", [False, True])
@pytest.mark.parametrize("n", [1, 2, 16, 31, 32, 33, 34, 1057, 1058])
@pytest.mark.parametrize("n_inst", [1, 33])
def test_queue_sizes_on_a_full_gpu(n_inst, n, equal):
    """The same with more than 20 warps per SM: every copy of a trace as the oracle."""
    B.build()
    cl = W.make_cluster(W.RECIPES[1])
    cl.inst_type = np.zeros(n_inst, np.uint8)
    cl.slots = np.array([1] * 3, np.int32)
    tr, grid, copies = _burst(n, equal, n), _grid([0]), 1600
    sim = H.Sim([tr] * copies, cl, grid)
    sim.run()
    got, want = sim.results(), oracle.run(W.Workload("queue", [tr], cl, grid, W.OBJ_P95))
    assert sim.info()["resident_warps"] > 20 * 152
    sim.close()
    for f in FIELDS:
        assert np.array_equal(got[f].reshape(copies, 2), np.tile(np.asarray(want[f]).reshape(1, 2), (copies, 1))), f


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["lean", "policies", "tenants", "faults"])
@pytest.mark.parametrize("n_inst", [8, 40])
def test_logged_budgets(n_inst, kind):
    name = {"tenants": "two-tenant", "faults": "faulty"}.get(kind)
    r = W.EXTRA[name] if name else W.RECIPES[1]
    tr = W.make_trace(r, 1, 3, n_queries=500)
    tr.arrival_us = tr.arrival_us // 4  # overdue requests: negative budgets
    cl = W.make_cluster(r)
    cl.inst_type = (np.arange(n_inst) % 3).astype(np.uint8)
    if cl.faults is not None:
        cl.faults["t0_us"] //= 4
        cl.faults["t1_us"] //= 4
    grid = _grid([0, 1, 2] if kind == "policies" else [0])
    assert _run(tr, cl, grid, record=list(range(grid.n_points))[::-1]) == 1


@pytest.mark.gpu
@pytest.mark.parametrize("recipe", [0, 4])
def test_far_first_query(recipe):
    """A trace whose first query lies 9.5 hours before the others: the same schedule
    and budgets as the oracle's, and the urgency keys cost the others no more than
    without the gap (deadlines that far overdue take exact 64-bit divisions, which
    is no business of requests that are not)."""
    wl = W.make_workload(recipe, n_traces=1, n_queries=1000)
    tr = wl.traces[0]
    gap = tr.arrival_us.copy()
    gap[1:] += 2 ** 35
    grid = W.subset_grid(wl.grid, [wl.grid.n_points - 1])  # alpha = 1: long queues
    cycles = []
    for t in (tr, W.Trace(**{**tr.__dict__, "arrival_us": gap})):
        _run(t, wl.cluster, grid, record=[0])
        sim = H.Sim([t], wl.cluster, grid)
        best = []
        for _ in range(7):
            sim.run()
            best.append(int(sim.results()["cycles_k"][0]))
        sim.close()
        cycles.append(min(best))
    assert cycles[1] < 1.1 * cycles[0], cycles
