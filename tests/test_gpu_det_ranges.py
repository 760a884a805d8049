"""Deterministic outcomes of a window whose rows are split over blocks: up to 76 outcomes in up to three groups of
32, and one more; scattered qubits, one and several column chunks."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,depth", [(200, 30), (2_100, 2), (5_000, 30)])
def test_repeated_windows(n, depth):
    c = C.random_circuit(n, depth, 0.5, seed=n, final_measure_all=False)
    q = np.random.default_rng(n).permutation(n)[:160].astype(np.uint32)
    sims = [qs.Simulator(n, flags=f) for f in (0, qs.QS_FLAG_NO_BLOCKED_MEASURE)]
    for sim in sims:
        sim.apply_layers_dev(sim.upload(c), 0, depth)
    first = [sim.measure(q, seed=1) for sim in sims]
    assert np.array_equal(*first)
    for count in (16, 32, 33, 64, 65, 76, 77, 152, 153):
        for sim in sims:
            assert np.array_equal(sim.measure(q[:count], seed=2), first[0][:count]), count
    sims[0].sync()
    assert not sims[0].record_kinds()[160:].any()
