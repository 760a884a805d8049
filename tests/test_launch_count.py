"""qs_sim_launch_count counts the kernels that a simulator's calls launch, on every path of the layers, the
measurements and the frame sampling."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from tests import fake_cuda
from workloads import circuits as C


@pytest.mark.parametrize("flags", [0, qs.QS_FLAG_NO_FUSION, qs.QS_FLAG_STEP_SYMBOLIC, qs.QS_FLAG_NO_BLOCKED_MEASURE,
                                   qs.QS_FLAG_INVERSE_TABLEAU])
@pytest.mark.parametrize("n", [1, 20, 256, 2_000, 17_000])
def test_count_is_the_launches(monkeypatch, n, flags):
    fake_cuda.use(monkeypatch)
    s = qs.qs_sim_create(n, flags=flags)
    sets = [C.random_circuit(n, d, 0.5, seed=1, final_measure_all=False) for d in (1, 2, 5, 40, 150)]
    sets.append(C.Circuit(n=n, gates=np.zeros((0, 3), np.uint32), layer_ptr=np.zeros(151, np.int64)))  # empty layers
    packed = [qs.qs_pack_layers(n, c.gates, c.layer_ptr) for c in sets]
    out = np.zeros(1 << 18, np.uint64)
    calls = [lambda c=c, p=p: qs.qs_sim_apply_layers_dev(s, p.ctypes.data, c.layer_ptr, 0, len(c.layer_ptr) - 1)
             for c, p in zip(sets, packed)]
    calls += [lambda m=m: qs.qs_sim_measure(s, np.arange(min(m, n)), 3) for m in (1, 15, 16, 64, 65, 500)]
    calls += [lambda: qs.qs_sim_apply_layer(s, sets[0].layer(0)), lambda: qs.qs_sim_noise(s, 0, 0.1, np.arange(n)),
              lambda: qs.qs_sim_measure(s, np.arange(min(n, 40)), 3), lambda: qs.qs_sim_tableau_export(s),
              lambda: qs.qs_sim_sample(s, 130, 1, out.ctypes.data, out.size), lambda: qs.qs_sim_reset(s)]
    assert qs.qs_sim_launch_count(s) == fake_cuda.count("launch")
    for i, f in enumerate(calls):
        f()
        assert qs.qs_sim_launch_count(s) == fake_cuda.count("launch"), i
    qs.qs_sim_destroy(s)
