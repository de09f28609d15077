"""Every family of the simulation kernel in its form for a full GPU, against the
oracle: one trace many times over, in more than one wave of warps, with per-call
logs, mixed policies, tenants and fault windows, with 32-bit and (one attempt
past 2^25 us) 64-bit times, with one and with two instances per lane; also on the
bounds-checked build."""
import numpy as np
import pytest

import oracle
from paper_2505_05286_gb300 import build as B
from paper_2505_05286_gb300 import hxsim as H
from paper_2505_05286_gb300 import workloads as W

pytestmark = pytest.mark.gpu
FIELDS = ["p95_us", "makespan_us", "events", "digest", "slo_met", "n_done", "status"]
EXTRAS = ["slo_met", "n_done", "reissued", "p95_us"]
KINDS = ["lean", "log", "policies", "tenants", "faults"]
COPIES, POINTS = 1600, 4


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def _inputs(kind, n_inst, long_calls):
    recipe = W.EXTRA["two-tenant"] if kind == "tenants" else W.RECIPES[1]
    tr = W.make_trace(recipe, 1, 90 + n_inst, n_queries=130)
    tr.arrival_us = tr.arrival_us // 5 // 200_000 * 200_000  # bursts that wait
    cl = W.make_cluster(recipe)
    cl.inst_type = (np.arange(n_inst) % 3).astype(np.uint8)
    cl.slots = np.array([1, 3, 16], np.int32)
    if kind == "faults":
        cl.timeout_mult_fp = 2 * W.SCALE
        cl.faults = np.zeros(3, W.FAULT_DTYPE)
        cl.faults[0] = (0, 0, 2_000_000, 6_000_000, 0)
        cl.faults[1] = (n_inst - 1, 0, 1_000_000, 9_000_000, 5 * W.SCALE)
        cl.faults[2] = (n_inst // 2, 0, 4_000_000, 5_000_000, W.SCALE // 2)
    if long_calls:
        tr.prompt[len(tr.prompt) // 2] = 1_000_000
    grid = W.Grid(np.array([0, W.SCALE // 3, W.SCALE, W.SCALE], np.int64),
                  np.array([W.SCALE, 0, 4 * W.SCALE, W.SCALE], np.int64), np.array([0, 1, 2, 15], np.int32),
                  np.full(POINTS, 300_000 ** 2, np.int64), np.zeros(POINTS, np.uint8), np.zeros(POINTS, np.uint8))
    if kind == "policies":
        grid.local_policy[:] = [W.POLICY_FCFS, W.POLICY_PQ, W.POLICY_FCFS, W.POLICY_LLF]
        grid.dispatch_policy[:2] = W.DISPATCH_RR
    return tr, cl, grid


def _check(kind, n_inst, long_calls, **kw):
    import torch
    tr, cl, grid = _inputs(kind, n_inst, long_calls)
    record = [1, POINTS * COPIES - 2, POINTS * (COPIES // 2)] if kind != "lean" else []
    sim = H.Sim([tr] * COPIES, cl, grid, record_sims=record, **kw)
    info = sim.info()
    full = 20 * torch.cuda.get_device_properties(0).multi_processor_count
    assert full < info["resident_warps"] < POINTS * COPIES  # not the few-warps form, and a second wave
    assert info["generic_kernel"] == int(long_calls or kind != "lean")
    sim.run()
    wl = W.Workload("full", [tr], cl, grid, W.OBJ_P95)
    want, extra = oracle.run(wl, range(POINTS), extra=True)
    got = sim.results()
    for f in FIELDS:
        assert np.array_equal(got[f].reshape(COPIES, POINTS), np.tile(np.asarray(want[f]), (COPIES, 1))), f
    got = sim.extras()
    for f in EXTRAS:
        assert np.array_equal(got[f].reshape(COPIES, -1), np.tile(np.asarray(extra[f]).reshape(1, -1), (COPIES, 1))), f
    for j, s in enumerate(record):
        _, log = oracle.simulate(tr, cl, oracle.point_of(grid, s % POINTS), log=True)
        lg = sim.records(j)
        for f in ("inst", "enq", "budget", "start", "end"):
            assert np.array_equal(lg[f], log[f]), (s, f)
    smem = info["smem_per_block"]
    sim.close()
    return smem


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n_inst", [1, 32, 33, 64])
def test_full_gpu_forms(n_inst, kind):
    # 64-bit times have slot entries of another size, by which they are told apart
    assert _check(kind, n_inst, False) != _check(kind, n_inst, True)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n_inst", [32, 64])
def test_full_gpu_forms_bounds_checked(n_inst, kind):
    H.load_checked()
    for long_calls in (False, True):
        _check(kind, n_inst, long_calls, bounds_checked=True)
