"""The simulation kernel's event loop at the edges of its representation, against
the oracle: times past 2^25, 2^31 and 2^32 us (with short calls event times are
32-bit, relative to a base that moves every 2^25 us), calls next to 2^25 us, calls
that end at the same time in one and in many slots, queries of more call records
than one sweep of the warp fetches."""
import numpy as np
import pytest

import oracle
from paper_2505_05286_gb300 import build as B
from paper_2505_05286_gb300 import hxsim as H
from paper_2505_05286_gb300 import workloads as W

FIELDS = ["p95_us", "makespan_us", "events", "digest", "slo_met", "n_done", "status"]
INST = [1, 16, 32, 33, 64]


def _workload(tr, cl, generic):
    B.build()
    n = 6
    lpol = (np.arange(n) % 3).astype(np.uint8) if generic else np.zeros(n, np.uint8)
    grid = W.Grid(np.array([0, W.SCALE // 7, W.SCALE // 2, W.SCALE * 6 // 7, W.SCALE, W.SCALE], np.int64),
                  np.array([W.SCALE, 0, 2 * W.SCALE, W.SCALE, W.SCALE // 4, 4 * W.SCALE], np.int64),
                  np.array([0, 1, 2, 3, 15, 0], np.int32), np.full(n, 300_000 ** 2, np.int64), lpol,
                  np.zeros(n, np.uint8))
    return W.Workload("core", [tr], cl, grid, W.OBJ_P95)


def _same(sim, wl, family):
    assert sim.info()["generic_kernel"] == int(family)
    sim.run()
    got, want = sim.results(), oracle.run(wl)
    for f in FIELDS:
        assert np.array_equal(got[f], want[f]), f


def _check(tr, cl, generic, family=None):
    wl = _workload(tr, cl, generic)
    sim = H.Sim(wl.traces, wl.cluster, wl.grid)
    _same(sim, wl, generic or cl.faults is not None if family is None else family)
    sim.close()


def _cluster(n_inst, slots=(1, 3, 16), rmax=2):
    cl = W.make_cluster(W.RECIPES[1])
    cl.inst_type = (np.arange(n_inst) % 3).astype(np.uint8)
    cl.slots = np.array(slots, np.int32)
    cl.rmax = rmax
    return cl


@pytest.mark.gpu
@pytest.mark.parametrize("long_calls", [False, True])
@pytest.mark.parametrize("kind", ["lean", "generic", "faults"])
@pytest.mark.parametrize("n_inst", INST)
def test_times_past_32_bits(n_inst, kind, long_calls):
    tr = W.make_trace(W.RECIPES[1], 1, 40 + n_inst, n_queries=160)
    # bursts at the edges of 25, 26, 31 and 32 bits and gaps of more than 2^32 us between
    # them, with calls of up to 20 s or 100 s running across
    at = np.array([0, 2 ** 25 - 1, 2 ** 25, 2 ** 26 - 1, 2 ** 26, 2 ** 31 - 10_000_000, 2 ** 31 - 1, 2 ** 31, 2 ** 32 - 3, 2 ** 32 + 2 ** 31 - 1,
                   3 * 2 ** 32 + 5, 9 * 2 ** 32 - 1], np.int64)
    tr.arrival_us = np.sort(np.concatenate([at + (i * 997) * (i % 5) for i in range(20)]))[:160]
    tr.prompt[::17] = 1_000_000 if long_calls else 100_000
    cl = _cluster(n_inst)
    if kind == "faults":
        cl.timeout_mult_fp = 2 * W.SCALE
        cl.faults = np.zeros(2, W.FAULT_DTYPE)
        cl.faults[0] = (0, 0, 2 ** 31 - 20_000_000, 2 ** 31 + 20_000_000, 0)
        cl.faults[1] = (n_inst - 1, 0, 2 ** 32 - 5, 2 ** 32 + 60_000_000, 4 * W.SCALE)
    _check(tr, cl, kind == "generic", long_calls or kind != "lean")


@pytest.mark.gpu
@pytest.mark.parametrize("n_inst", [32, 33])
def test_calls_next_to_the_short_limit(n_inst):
    """Calls of 2^25 - 1 us keep 32-bit times, 2^25 us take 64-bit ones; a handle
    follows the traces it is given, in either direction."""
    cl = _cluster(n_inst)
    cl.prefill_tok_s[:] = 1_000_000
    cl.decode_us_tok[:] = 32
    short = W.make_trace(W.RECIPES[1], 1, 9, n_queries=100)
    short.prompt[:] = 1 + short.prompt % 900_000
    short.prompt[::3], short.out[::3], short.out_est[::3] = 31, (2 ** 20 - 1), (2 ** 20 - 1)
    assert int((short.prompt.astype(np.int64) + 32 * np.maximum(short.out, short.out_est)).max()) == 2 ** 25 - 1
    longer = W.Trace(short.arrival_us, short.k, short.call_base, short.prompt.copy(), short.out, short.out_est,
                     short.stage, short.cand, short.retry)
    longer.prompt[::3] = 32
    a, b = _workload(short, cl, False), _workload(longer, cl, False)
    sim = H.Sim(a.traces, cl, a.grid)
    _same(sim, a, 0)
    sim.upload(b.traces)
    _same(sim, b, 1)
    sim.upload(a.traces)
    _same(sim, a, 0)
    sim.close()
    sim = H.Sim(b.traces, cl, b.grid)
    _same(sim, b, 1)
    sim.close()
    for wl in (a, b):
        got, _ = H.run_static(wl.traces[0], cl, wl.grid)
        assert np.array_equal(got["digest"], oracle.run(wl)["digest"])


@pytest.mark.gpu
@pytest.mark.parametrize("n_inst", [3, 40])
@pytest.mark.parametrize("slow,timeout", [(2, 0), (2, 2), (0.5, 1), (0, 2), (100, 0)])
def test_attempts_next_to_the_short_limit(n_inst, slow, timeout):
    """Fault windows whose slow-down or timeout takes a call to 2^25 - 1, 2^25 and
    past it: the same results with 32-bit and with 64-bit times."""
    cl = _cluster(n_inst)
    cl.prefill_tok_s[:] = 1_000_000
    cl.decode_us_tok[:] = 32
    cl.timeout_mult_fp = timeout * W.SCALE
    cl.faults = np.zeros(2, W.FAULT_DTYPE)
    cl.faults[0] = (0, 0, 0, 400_000_000, int(slow * W.SCALE))
    cl.faults[1] = (n_inst - 1, 0, 100_000_000, 600_000_000, W.SCALE)
    stretch = max(slow, timeout, 1)
    for cost in (2 ** 25 // stretch - 1, 2 ** 25 // stretch, 2 ** 25 // stretch + 2):
        tr = W.make_trace(W.RECIPES[1], 1, 21, n_queries=60)
        tr.arrival_us = tr.arrival_us * 20
        tr.out[::2] = tr.out_est[::2] = int(cost) // 32 - 1
        tr.prompt[::2] = int(cost) - 32 * (int(cost) // 32 - 1)
        _check(tr, cl, True, 1)


@pytest.mark.gpu
@pytest.mark.parametrize("n_inst,on", [(1, [0]), (32, [31]), (32, list(range(16))), (33, [32]), (64, [0, 31, 32, 63]), (64, [])])
def test_windows_of_some_instances(n_inst, on):
    """Instances without fault windows beside ones that have some (at the edges of
    a lane's first and second), and windows that no call meets."""
    cl = _cluster(n_inst)
    cl.timeout_mult_fp = 2 * W.SCALE
    cl.faults = np.zeros(len(on) or 1, W.FAULT_DTYPE)
    cl.faults[0] = (0, 0, 2 ** 37, 2 ** 38, W.SCALE)
    for i, m in enumerate(on):
        cl.faults[i] = (m, 0, 5_000_000 * i, 40_000_000 + 5_000_000 * i, (3 * W.SCALE, 0)[i % 2])
    tr = W.make_trace(W.RECIPES[1], 1, 80 + n_inst, n_queries=120)
    _check(tr, cl, True, 1)


@pytest.mark.gpu
@pytest.mark.parametrize("generic", [False, True])
@pytest.mark.parametrize("slots", [(1, 1, 1), (16, 16, 16), (2, 15, 16)])
@pytest.mark.parametrize("n_inst", INST)
def test_equal_completion_times(n_inst, slots, generic):
    tr = W.make_trace(W.RECIPES[1], 1, 60 + n_inst, n_queries=120)
    tr.prompt[:] = 2000
    tr.out[:] = 100
    tr.out_est[:] = 100
    tr.arrival_us = (np.arange(120) // 15 * 400_000).astype(np.int64)
    _check(tr, _cluster(n_inst, slots), generic)


@pytest.mark.gpu
@pytest.mark.parametrize("n_inst", [4, 64])
def test_queries_of_many_calls(n_inst):
    r = W.Recipe(**{**W.EXTRA["paper-shaped"].__dict__, "p_err": 0.97, "rmax": 15})
    tr = W.make_trace(r, 17, 5, n_queries=40)
    assert int(np.diff(tr.call_base).max()) > 64
    _check(tr, _cluster(n_inst, rmax=15), False)
