"""Short fused segments: layers of one and of several gates a thread, beyond the records of the ring
(more than 4,096 gates), fewer layers than ring stages, and columns that leave no room for the ring."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,layers", [(1, 4), (100, 7), (1_100, 9), (1_300, 8), (5_500, 4), (5_950, 4), (14_080, 4)])
def test_short_segments_equal_single_layers(n, layers):
    c = C.gate_mix_circuit(n, layers, seed=n, final_measure_all=False)
    q = np.arange(0, n, max(1, n // 40), dtype=np.uint32)
    circ = C.Circuit(n=n, gates=c.gates, layer_ptr=c.layer_ptr, ops=[("layers", 0, layers), ("measure", q)])
    out = []
    for flags in (0, qs.QS_FLAG_NO_FUSION):
        sim = qs.Simulator(n, flags=flags)
        rec = sim.run(circ, seed=3, dc=sim.upload(circ))
        out.append([rec, qs.qs_sim_tableau_export(sim.sim), sim.sample(300, seed=9, on_device=False)])
        sim.sync()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
