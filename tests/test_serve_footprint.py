"""The serving loop's admission counts what a request holds on the device when it runs in a batch."""
import ctypes

import numpy as np
import pytest

from paper_2603_14641_gb300 import qs, serve
from workloads import circuits as C


@pytest.mark.parametrize("n", [5, 100, 640, 641, 800, 1_023])
@pytest.mark.parametrize("shots", [1, 10_000])
def test_footprint_covers_a_batched_request(n, shots):
    c = C.random_circuit(n, 30, 0.5, seed=1)
    ex = serve.GpuExecutor.__new__(serve.GpuExecutor)  # no device here
    ex.qs = qs
    req = serve.Request(0, 0.0, c, shots, seed=1)
    g, lp = np.ascontiguousarray(c.gates, np.uint32), np.ascontiguousarray(c.layer_ptr, np.int64)
    rl, rm, q = qs.circuit_rounds(c)
    arr = (qs.qs_batch_circuit * 1)(qs.qs_batch_circuit(n, c.n_layers, g.ctypes.data, lp.ctypes.data, len(rl) - 1, 0,
                                                        rl.ctypes.data, rm.ctypes.data, q.ctypes.data, 1, 0))
    assert ex.batchable(req)
    batch = qs.lib().qs_batch_required_bytes(1, ctypes.byref(arr))
    sim = qs.qs_sim_required_bytes(n, record_capacity=c.n_measurements) if n > 640 else 0
    samples = c.n_measurements * ((shots + 63) // 64) * 8
    assert ex.batch_footprint(req) >= batch + sim + samples


def test_a_batch_counts_all_its_members_so():
    """Alone a request of 60 fits a budget of 100; in a batch it takes 90, and two batched ones of 45 fit."""
    sizes, seen = {0: (60, 90), 1: (60, 90), 2: (30, 45), 3: (30, 45), 4: (30, 60), 5: (30, 30)}, []

    def run(req, slot, admit, fp):
        seen.append(([req.rid], [fp]))
        return serve.Result(req.rid, 0, 0, 0.0, admit, 0.0, fp)

    def run_batch(reqs, slot, admit, fps):
        seen.append(([r.rid for r in reqs], list(fps)))
        return [serve.Result(r.rid, 0, 0, 0.0, admit, 0.0, f) for r, f in zip(reqs, fps)]

    sch = serve.Scheduler(1, 100, lambda r: sizes[r.rid][0], run, execute_batch=run_batch, batchable=lambda r: True,
                          batch_footprint=lambda r: sizes[r.rid][1])
    for i in range(6):
        sch.pending.append(serve.Request(i, 0.0, None, 0, i))
    sch.run([])
    assert seen == [([0], [60]), ([1], [60]), ([2, 3], [45, 45]), ([4, 5], [60, 30])]
    assert sch.in_use == 0 and sch.peak_in_use == 90
