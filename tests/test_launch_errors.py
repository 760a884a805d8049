"""A launch that fails makes the call fail, wherever in a window it is and whether or not kernel classes are
timed meanwhile (event queries in between must not lose it)."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from tests import fake_cuda
from workloads import circuits as C


@pytest.mark.parametrize("n,flags", [(4_096 + 200, 0), (300, qs.QS_FLAG_INVERSE_TABLEAU), (300, qs.QS_FLAG_STEP_SYMBOLIC)])
@pytest.mark.parametrize("timed", [False, True])
def test_measurement_window(monkeypatch, n, flags, timed):
    L = fake_cuda.use(monkeypatch)
    q = np.arange(n, dtype=np.uint32)

    def window(fail):
        s = qs.qs_sim_create(n, flags=flags)
        if timed:
            qs.qs_sim_set_timing(s, True)
        qs.qs_sim_measure(s, q[:1], 1)  # the layout switch is done
        L.fake_reset(fail, 1)
        qs.qs_sim_measure(s, q, 3, want_outcomes=False)
        return s

    s = window(-1)
    launches = fake_cuda.count("launch")
    L.fake_reset(-1, 0)
    qs.qs_sim_destroy(s)
    for fail in {0, 1, 2, 3, 5, launches // 2, launches - 2, launches - 1}:
        with pytest.raises(qs.QsError) as e:
            window(fail)
        assert e.value.code == -3, fail
        assert L.cudaGetLastError() == 0, "an error was left for a later call"


def test_layers_and_samples(monkeypatch):
    L = fake_cuda.use(monkeypatch)
    out = np.zeros(1 << 20, np.uint64)
    for n, flags in ((200, 0), (200, qs.QS_FLAG_NO_FUSION), (2_000, 0), (200, qs.QS_FLAG_INVERSE_TABLEAU)):
        c = C.gate_mix_circuit(n, 40, seed=1, final_measure_all=False)
        packed = qs.qs_pack_layers(n, c.gates, c.layer_ptr)
        fail = 0
        while True:
            L.fake_reset(-1, 0)
            s = qs.qs_sim_create(n, flags=flags)
            L.fake_reset(fail, 0)
            try:
                qs.qs_sim_apply_layers_dev(s, packed.ctypes.data, c.layer_ptr, 0, 40)
                qs.qs_sim_apply_layer(s, c.layer(0))
                qs.qs_sim_noise(s, qs.QS_NOISE_X, 0.1, np.arange(n))
                qs.qs_sim_measure(s, np.arange(3), 1)
                qs.qs_sim_sample(s, 100, 1, out.ctypes.data, out.size)
            except qs.QsError as e:
                assert e.code == -3 and L.cudaGetLastError() == 0
            else:
                assert fail >= fake_cuda.count("launch") > 5
                break
            fail += 1
