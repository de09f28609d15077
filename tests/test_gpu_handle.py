"""What a handle reserves on the device and the host, and which kernels it runs."""
import ctypes
import time

import numpy as np
import pytest

import oracle
from paper_2505_05286_gb300 import build as B
from paper_2505_05286_gb300 import hxsim as H
from paper_2505_05286_gb300 import workloads as W

pytestmark = pytest.mark.gpu
FIELDS = ["p95_us", "makespan_us", "events", "digest", "slo_met", "n_done", "status"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def test_arena_holds_no_more_than_a_queue_offset_reaches():
    """A local queue's place in the arena is kept in 27 bits: entries past 2^27 a
    warp could not be told from others, so a handle takes none."""
    wl = W.make_workload(0, n_queries=20)
    scratch = []
    for entries in (2 ** 27, 2 ** 27 + 1000):
        sim = H.Sim(wl.traces, wl.cluster, wl.grid, max_resident_warps=4, arena_entries=entries)
        scratch.append(sim.info()["scratch_bytes"])
        sim.run()
        got, want = sim.results(), oracle.run(wl)
        sim.close()
        for f in FIELDS:
            assert np.array_equal(got[f], want[f]), f
    assert scratch[0] == scratch[1] > 4 * 16 * 2 ** 27


def _logged(queries):
    """A run of two traces of these queries and of half as many with every call of both logged."""
    wl = W.make_workload(4, n_traces=1, n_queries=queries)
    wl.traces.append(W.make_workload(4, n_traces=2, n_queries=queries // 2).traces[1])
    wl.grid = W.subset_grid(wl.grid, [0])
    sim = H.Sim(wl.traces, wl.cluster, wl.grid, record_sims=[1, 0])
    sim.run()
    return wl, sim


@pytest.mark.parametrize("queries", [40, 380, 420, 1580, 1620, 5000])  # 300 to 38000 calls
def test_records_by_column(queries):
    """Any choice of the log's columns, read in one copy (short logs) or by column."""
    wl, sim = _logged(queries)
    names = ("inst", "enq", "budget", "start", "end")
    for j, t in enumerate((1, 0)):
        _, want = oracle.simulate(wl.traces[t], wl.cluster, oracle.point_of(wl.grid, 0), log=True)
        n = len(wl.traces[t].prompt)
        for pick in (names, ("end",), ("inst",), ("enq", "budget"), ("inst", "start", "end")):
            out = {f: np.full(n, -7, np.int32 if f == "inst" else np.int64) for f in names}
            assert sim.lib.hx_sim_records(sim.h, j, *[H._p(out[f]) if f in pick else None for f in names], n) == H.HX_OK
            for f in names:
                assert np.array_equal(out[f], want[f]) if f in pick else (out[f] == -7).all(), (pick, f)
    sim.close()


def test_one_column_of_a_long_log_costs_one_copy():
    """Reading one column of 150k calls takes about as long as a copy of its bytes
    (five times that when the whole log went through a buffer)."""
    import torch
    wl, sim = _logged(20000)
    n = len(wl.traces[0].prompt)
    host, dev = torch.zeros(n, dtype=torch.int64), torch.zeros(n, dtype=torch.int64, device="cuda")
    at = ctypes.c_void_p(host.data_ptr())

    def median_us(read):
        t = []
        for _ in range(41):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            read()
            t.append(1e6 * (time.perf_counter() - t0))
        return sorted(t)[20]
    column = median_us(lambda: sim.lib.hx_sim_records(sim.h, 1, None, None, None, None, at, n))
    copy = median_us(lambda: host.copy_(dev))
    sim.close()
    assert column < 2.5 * copy + 10, (column, copy)


class _MallInfo(ctypes.Structure):
    _fields_ = [(f, ctypes.c_size_t) for f in ("arena", "ordblks", "smblks", "hblks", "hblkhd", "usmblks", "fsmblks",
                                               "uordblks", "fordblks", "keepcost")]


def _host_bytes():
    """Bytes that malloc has handed out (main arena and mapped blocks)."""
    info = ctypes.CDLL(None).mallinfo2
    info.restype = _MallInfo
    m = info()
    return m.uordblks + m.hblkhd


@pytest.mark.parametrize("n,queries,staged", [(1, 11000, True), (1, 12000, False), (2, 30000, False), (8, 20000, True)])
def test_calls_are_staged_where_that_is_cheaper(n, queries, staged):
    """A handle keeps a host copy of its calls only where one copy of it is cheaper
    than copies of every trace's arrays: not for a few large traces."""
    wl = W.make_workload(1, n_traces=n, n_queries=queries)
    wl.grid = W.subset_grid(wl.grid, [5])
    H.Sim(wl.traces, wl.cluster, wl.grid, max_resident_warps=4).close()
    before = _host_bytes()
    sim = H.Sim(wl.traces, wl.cluster, wl.grid, max_resident_warps=4)
    kept = _host_bytes() - before
    per_call = 15 * sum(len(t.prompt) for t in wl.traces)
    assert (kept > per_call) == staged, (kept, per_call)
    for step in range(2):  # a new handle's inputs, and an upload's
        sim.run()
        got, want = sim.results(), oracle.run(wl)
        for f in FIELDS:
            assert np.array_equal(got[f], want[f]), f
        sim.upload(wl.traces)
    sim.close()


@pytest.mark.parametrize("record", [(), (4097,)])
@pytest.mark.parametrize("n", [1, 5, 100])
def test_a_subset_is_sized_by_what_runs(n, record):
    """A few simulations of a large grid take the warps and the scratch that they
    need (and with them the kernels for runs of few warps), not the grid's."""
    wl = W.make_workload(2, n_traces=32, n_queries=60)
    subset = [4097 + 13 * i for i in range(n)]
    sim = H.Sim(wl.traces, wl.cluster, wl.grid, subset=subset, record_sims=record)
    info = sim.info()
    assert info["blocks"] == -(-n // info["warps_per_block"])
    few = H.Sim(wl.traces, wl.cluster, W.subset_grid(wl.grid, [0]), max_resident_warps=4)
    assert info["scratch_bytes"] == info["blocks"] * few.info()["scratch_bytes"]
    few.close()
    sim.run()
    got, want = sim.results(), oracle.run(wl, subset)
    sim.close()
    for f in FIELDS:
        assert np.array_equal(got[f][subset], want[f]), f
    assert (np.delete(got["status"], subset) == H.HX_SKIPPED).all()


@pytest.mark.parametrize("n_inst", [8, 32])
def test_long_calls_keep_a_full_gpu(n_inst):
    """A call past 2^25 us moves the whole run to 64-bit times: its slots then take
    twice the room, which must not cost the run more than a block an SM."""
    wl = W.make_workload(1, n_traces=80, n_queries=20)
    wl.cluster.inst_type = (np.arange(n_inst) % 3).astype(np.uint8)  # 4 to 16 slots each
    sim = H.Sim(wl.traces, wl.cluster, wl.grid)
    short = sim.info()["blocks"]
    sim.close()
    wl.traces[3].prompt[7] = 1_000_000
    sim = H.Sim(wl.traces, wl.cluster, wl.grid)
    assert sim.info()["generic_kernel"] == 1 and sim.info()["blocks"] >= short * 7 // 8
    sim.run()
    got, want = sim.results(), oracle.run(wl)
    sim.close()
    for f in FIELDS:
        assert np.array_equal(got[f], want[f]), f


@pytest.mark.parametrize("n_inst", [3, 40])
@pytest.mark.parametrize("slow,timeout", [(None, 0), (2, 0), (2, 2), (0.5, 1), (0, 2), (3, 7), (100, 0)])
def test_times_are_64_bit_only_where_an_attempt_needs_them(n_inst, slow, timeout):
    """The first attempt length (slowed or timed out by the fault windows) that takes
    64-bit times is 2^25 us; told by the room that a block's slot entries take."""
    wl = W.make_workload(1, n_traces=1, n_queries=5)
    tr, cl = wl.traces[0], wl.cluster
    cl.inst_type = (np.arange(n_inst) % 3).astype(np.uint8)
    cl.prefill_tok_s[:], cl.decode_us_tok[:] = 1_000_000, 32
    stretch = W.SCALE
    if slow is not None:
        cl.timeout_mult_fp = timeout * W.SCALE
        cl.faults = np.zeros(1, W.FAULT_DTYPE)
        cl.faults[0] = (n_inst - 1, 0, 0, 1000, int(slow * W.SCALE))
        stretch = max(stretch, cl.timeout_mult_fp, int(slow * W.SCALE))
    first = (2 ** 25 - 1) * W.SCALE // stretch + 1  # us of the shortest such call

    def smem(cost):
        tr.prompt[:], tr.out[:], tr.out_est[:] = 1, 1, 1
        tr.out[3] = (cost - 1) // 32
        tr.prompt[3] = cost - 32 * int(tr.out[3])
        sim = H.Sim([tr], cl, wl.grid)
        block = sim.info()["smem_per_block"]
        sim.close()
        return block
    assert smem(first - 1) == smem(first // 2)
    assert smem(first) == smem(first + 1) > smem(first - 1)
