"""Fused gate segments at the edges of their slices: words per block from 1 to 8, 32-bit slices, runs
longer than one set of records (128 layers), and the shortest run that is fused (4 layers)."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


def _both(circ, shots):
    out = []
    for flags in (0, qs.QS_FLAG_NO_FUSION):
        sim = qs.Simulator(circ.n, flags=flags)
        dc = sim.upload(circ)
        rec = sim.run(circ, seed=3, dc=dc)
        out.append([rec, qs.qs_sim_tableau_export(sim.sim)] + [sim.sample(s, seed=9, on_device=False) for s in shots])
        sim.sync()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [1, 2, 9, 63, 64, 130])
def test_frame_slices_of_every_width(n):
    """Shot words 1, 2, 3, 4, 5, 8, 9, 31 and enough for several blocks of 8 words per SM."""
    c = C.gate_mix_circuit(n, 13, seed=n, measure_every=6, measure_frac=0.5)
    _both(c, [1, 64, 130, 256, 257, 512, 513, 1_970, 64 * 9_731 + 5])


@pytest.mark.parametrize("n,layers", [(40, 300), (257, 129), (700, 128), (5_000, 4), (5_000, 3), (9_999, 5)])
def test_long_and_short_runs(n, layers):
    """Runs across the 128-layer limit and around the 4-layer threshold, with an empty layer."""
    c = C.gate_mix_circuit(n, layers, seed=layers, final_measure_all=False)
    lp = np.concatenate([c.layer_ptr[:2], c.layer_ptr[1:]])
    ops = [("layers", 0, len(lp) - 1), ("measure", np.arange(0, n, max(1, n // 50), dtype=np.uint32))]
    _both(C.Circuit(n=n, gates=c.gates, layer_ptr=lp, ops=ops), [64, 700])


def test_invalid_device_records_are_skipped_and_reported():
    """A record with an unknown type or a qubit out of range changes nothing and fails the next sync."""
    import torch
    for bad in ((13 << 24, 0), (C.H << 24 | 40, 0), (C.CX << 24 | 1, 40), (C.CX << 24 | 3, 3)):
        for n_layers in (2, 6):
            sim = qs.Simulator(40)
            rec = np.zeros((n_layers, 2), np.uint32)
            rec[:, 0] = C.X << 24 | 5
            rec[1] = bad
            dev = torch.from_numpy(rec.view(np.int32)).cuda()
            qs.qs_sim_apply_layers_dev(sim.sim, dev.data_ptr(), np.arange(n_layers + 1), 0, n_layers)
            with pytest.raises(qs.QsError) as e:
                sim.sync()
            assert e.value.code == -7
