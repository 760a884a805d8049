"""Host code of the simulators on a CUDA runtime without a GPU: what creating one allocates."""
import numpy as np

from paper_2603_14641_gb300 import qs
from tests import fake_cuda
from workloads import circuits as C


def test_pinned_slots_come_with_their_first_use(monkeypatch):
    """Creating a simulator and running device lists pins no host memory; staged calls take up to four slots,
    and a simulator with all of them goes on."""
    fake_cuda.use(monkeypatch)
    n = 3_000
    s = qs.qs_sim_create(n)
    c = C.random_circuit(n, 6, 0.5, seed=1, final_measure_all=False)
    packed = qs.qs_pack_layers(n, c.gates, c.layer_ptr)
    qs.qs_sim_apply_layers_dev(s, packed.ctypes.data, c.layer_ptr, 0, 6)
    qs.qs_sim_measure(s, np.arange(100), 1)
    assert fake_cuda.count("pinned") == 0
    for i in range(6):
        qs.qs_sim_reset(s, np.ones(n, np.uint8))
        assert fake_cuda.count("pinned") == min(i + 1, 4)
    qs.qs_sim_destroy(s)
