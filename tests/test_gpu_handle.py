"""What a handle reserves on the device and the host, and which kernels it runs."""
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
