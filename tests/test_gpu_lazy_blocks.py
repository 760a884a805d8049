"""Runs of layers with deferred one-qubit gates, in blocks whose last warp is not whole (252, 220 and 222
threads) and in whole ones: equal to the same layers one call each, where no gate is deferred."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,flags", [(2, 1), (64, 1), (700, 1), (2_800, 1), (14_081, 0), (16_400, 0)])
def test_runs_equal_single_layers(n, flags):
    c = C.gate_mix_circuit(n, 6, seed=n, final_measure_all=False)
    packed = qs.qs_pack_layers(n, c.gates, c.layer_ptr).view(np.int32)
    out = []
    for step, shift in ((6, 0), (1, 0), (6, 1)):  # shift: records at 4 bytes
        sim = qs.Simulator(n, flags=flags)
        dev = torch.zeros(len(packed) + 1, dtype=torch.int32, device="cuda")
        dev[shift:shift + len(packed)] = torch.from_numpy(packed).cuda()
        for l in range(0, 6, step):
            qs.qs_sim_apply_layers_dev(sim.sim, dev.data_ptr() + 4 * shift, c.layer_ptr, l, l + step)
        out.append(qs.qs_sim_tableau_export(sim.sim))
        sim.sync()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
