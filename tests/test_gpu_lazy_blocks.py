"""Runs of layers with deferred one-qubit gates, in blocks whose last warp is not whole (252, 220 and 222
threads) and in whole ones: equal to the same layers one call each, where no gate is deferred."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,flags", [(2, 1), (64, 1), (700, 1), (2_800, 1), (14_081, 0), (16_400, 0)])
def test_runs_equal_single_layers(n, flags):
    c = C.gate_mix_circuit(n, 6, seed=n, final_measure_all=False)
    out = []
    for step in (6, 1):
        sim = qs.Simulator(n, flags=flags)
        dc = sim.upload(c)
        for l in range(0, 6, step):
            sim.apply_layers_dev(dc, l, l + step)
        out.append(qs.qs_sim_tableau_export(sim.sim))
        sim.sync()
    assert np.array_equal(*out)
