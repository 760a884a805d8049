"""A reset writes the whole state: small tableaus in one launch, larger ones by memsets and kernels."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 65, 300, 5_632, 5_800])
@pytest.mark.parametrize("flags", [0, qs.QS_FLAG_INVERSE_TABLEAU])
def test_reset_after_use_equals_a_basis_state(n, flags):
    sim = qs.Simulator(n, flags=flags)
    sim.run(C.gate_mix_circuit(n, 4, seed=n, final_measure_all=False), seed=1)
    sim.measure(np.arange(min(n, 20), dtype=np.uint32), seed=2)
    init = (np.arange(n) % 3 == 1).astype(np.uint8)
    sim.reset(init)
    x, z, r = sim.export()
    eye = np.eye(n, dtype=bool)
    assert np.array_equal(np.asarray(x, bool), np.vstack([eye, np.zeros((n, n), bool)]))
    assert np.array_equal(np.asarray(z, bool), np.vstack([np.zeros((n, n), bool), eye]))
    if not flags:
        assert np.array_equal(np.asarray(r, np.uint8), np.concatenate([init, init]))
    assert sim.num_measurements == 0
    assert np.array_equal(sim.measure(np.arange(n, dtype=np.uint32), seed=3), init)
    sim.sync()
