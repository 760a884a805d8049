"""Paths against arms that share none of their code: fused segments against layers one call each, and the symbolic
pass of a block above 16,384 qubits (256 rows a block) against one launch per step."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,depth", [(300, 130), (2_500, 40), (5_000, 40), (14_080, 20)])
def test_fused_segments_equal_layers_one_call_each(n, depth):
    c = C.gate_mix_circuit(n, depth, seed=n, final_measure_all=False)
    out = []
    for step in (depth, 1):
        sim = qs.Simulator(n)
        dc = sim.upload(c)
        for l in range(0, depth, step):
            sim.apply_layers_dev(dc, l, l + step)
        out.append(qs.qs_sim_tableau_export(sim.sim))
        sim.measure(np.arange(0, n, 7, dtype=np.uint32), seed=2)
        out.append(sim.sample(600, 5, on_device=False))
        sim.sync()
    assert np.array_equal(out[0], out[2]) and np.array_equal(out[1], out[3])


def test_step_symbolic_pass_of_a_large_tableau():
    n = 17_000
    c = C.random_circuit(n, 5, 0.4, seed=3, final_measure_all=False)
    q = np.random.default_rng(1).permutation(n)[:90].astype(np.uint32)
    q[70:80] = q[:10]
    out = []
    for flags in (0, qs.QS_FLAG_STEP_SYMBOLIC):
        sim = qs.Simulator(n, flags=flags)
        sim.apply_layers_dev(sim.upload(c), 0, 5)
        rec = sim.measure(q, seed=4)
        out.append((rec, sim.record_kinds(), qs.qs_sim_tableau_export(sim.sim)))
        sim.sync()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    assert 0 < out[0][1].sum() < len(q)
