"""The dispatcher's choice of instance (Eq. score) on the GPU: the float filter
and the exact path it falls back to, against the oracle, where bounds overlap or
scores tie: equal instances, rewards of 0 or at the cap, alpha next to 0 and 1,
clusters at the edges of one and two instances per lane."""
import numpy as np
import pytest

import oracle
from paper_2505_05286_gb300 import build as B
from paper_2505_05286_gb300 import hxsim as H
from paper_2505_05286_gb300 import workloads as W

FIELDS = ["p95_us", "makespan_us", "events", "digest", "slo_met", "n_done", "status"]
ALPHAS = [0, 1, W.SCALE // 2, W.SCALE - 1, W.SCALE]
BETAS = [0, 1, 2 ** 20, 300_000 ** 2, 2 ** 43, 2 ** 62]


def _grid(generic):
    a, b = [x.ravel() for x in np.meshgrid(ALPHAS, BETAS, indexing="ij")]
    n = a.size
    lpol = (np.arange(n) % 3).astype(np.uint8) if generic else np.zeros(n, np.uint8)
    return W.Grid(a.astype(np.int64), np.full(n, W.SCALE, np.int64), np.full(n, 2, np.int32), b.astype(np.int64),
                  lpol, np.zeros(n, np.uint8))


@pytest.mark.gpu
@pytest.mark.parametrize("generic", [False, True])
@pytest.mark.parametrize("n_inst", [1, 2, 31, 32, 33, 63, 64])
@pytest.mark.parametrize("types", ["one", "near", "mixed"])
def test_winner_matches_the_oracle(types, n_inst, generic):
    B.build()
    r = W.RECIPES[1]
    tr = W.make_trace(r, 1, 7 + n_inst, n_queries=300)
    tr.arrival_us = tr.arrival_us // 8  # queues and idle instances both occur
    cl = W.make_cluster(r)
    # "near": costs one microsecond per token apart, far below the rewards' float spacing
    prof = {"one": [(12000, 15)], "near": [(12000, 15), (12001, 15), (12000, 16)],
            "mixed": [(5000, 35), (9000, 22), (12000, 15), (20000, 10)]}[types]
    cl.prefill_tok_s = np.array([p for p, _ in prof], np.int32)
    cl.decode_us_tok = np.array([d for _, d in prof], np.int32)
    cl.slots = np.array([3, 1, 2, 16][:len(prof)], np.int32)
    cl.inst_type = (np.arange(n_inst) % len(prof)).astype(np.uint8)
    cl.ref_type = 0
    wl = W.Workload("dispatch", [tr], cl, _grid(generic), W.OBJ_P95)
    sim = H.Sim(wl.traces, wl.cluster, wl.grid)
    assert sim.info()["generic_kernel"] == int(generic)
    sim.run()
    got, want = sim.results(), oracle.run(wl)
    sim.close()
    for f in FIELDS:
        assert np.array_equal(got[f], want[f]), f
