"""Which runs of device layers are fused or have their one-qubit gates deferred, by the launches they take: one
each, one for a short fused run, and the layers plus two where gates are deferred."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from tests import fake_cuda
from workloads import circuits as C


def _launches(sim, c, layers):
    packed = qs.qs_pack_layers(c.n, c.gates, c.layer_ptr)
    before = fake_cuda.count("launch")
    qs.qs_sim_apply_layers_dev(sim, packed.ctypes.data, c.layer_ptr, 0, layers)
    return fake_cuda.count("launch") - before


@pytest.mark.parametrize("n,p,layers,launches", [
    (256, 0.5, 1, 1), (256, 0.5, 2, 1), (1_024, 0.5, 3, 1), (1_025, 0.5, 3, 3), (1_025, 0.5, 4, 1),
    (14_500, 0.5, 2, 2), (14_500, 0.5, 3, 3), (14_500, 0.5, 4, 6), (20_000, 0.8, 3, 3), (25_000, 0.5, 2, 2),
    (25_000, 0.5, 3, 5), (41_000, 0.5, 2, 4),
    (14_500, 1.0, 8, 8), (14_501, 1.0, 8, 8), (14_500, 0.0, 4, 6)])
def test_runs(monkeypatch, n, p, layers, launches):
    fake_cuda.use(monkeypatch)
    s = qs.qs_sim_create(n)
    assert _launches(s, C.random_circuit(n, layers, p, seed=1, final_measure_all=False), layers) == launches
    qs.qs_sim_destroy(s)


def test_a_layer_of_one_qubit_gates_among_pairs(monkeypatch):
    """H on every qubit and layers of pairs: deferred if a third of the layers may hold one-qubit gates."""
    fake_cuda.use(monkeypatch)
    n = 15_000
    s = qs.qs_sim_create(n)
    h = np.stack([np.full(n, C.H), np.arange(n), np.zeros(n)], 1).astype(np.uint32)
    cz = np.stack([np.full(n // 2, C.CZ), np.arange(0, n, 2), np.arange(1, n, 2)], 1).astype(np.uint32)
    for order, deferred in (("HCHC", True), ("HCCHCC", True), ("HCCCHCCC", False), ("C.C.C.H.H.", True), ("H..C.", False)):
        gates = [{"H": h, "C": cz, ".": h[:0]}[k] for k in order]
        lp = np.cumsum([0] + [len(g) for g in gates])
        c = C.Circuit(n=n, gates=np.concatenate(gates), layer_ptr=lp, ops=[])
        full = sum(len(g) > 0 for g in gates)
        assert _launches(s, c, len(gates)) == full + 2 * deferred, order
    qs.qs_sim_destroy(s)


def test_records_at_four_bytes_are_not_fused(monkeypatch):
    fake_cuda.use(monkeypatch)
    c = C.random_circuit(300, 5, 0.5, seed=1, final_measure_all=False)
    packed = np.zeros(2 * len(c.gates) + 1, np.uint32)
    packed[1:] = qs.qs_pack_layers(300, c.gates, c.layer_ptr)
    s = qs.qs_sim_create(300)
    for shift, launches in ((0, 1), (4, 5)):
        before = fake_cuda.count("launch")
        qs.qs_sim_apply_layers_dev(s, packed.ctypes.data + shift, c.layer_ptr, 0, 5)
        assert fake_cuda.count("launch") - before == launches
    qs.qs_sim_destroy(s)


@pytest.mark.gpu
def test_runs_equal_layers_one_call_each():
    """The shortest fused runs, and records at four bytes."""
    import torch
    for n, layers in ((2, 2), (256, 3), (1_024, 2), (1_025, 3), (300, 5)):
        c = C.gate_mix_circuit(n, layers, seed=n, final_measure_all=False)
        packed = qs.qs_pack_layers(n, c.gates, c.layer_ptr).view(np.int32)
        dev = [torch.zeros(len(packed) + 1, dtype=torch.int32, device="cuda") for _ in range(2)]
        out = []
        for shift, step in ((0, layers), (0, 1), (1, layers)):
            dev[shift][shift:shift + len(packed)] = torch.from_numpy(packed).cuda()
            sim = qs.Simulator(n)
            for l in range(0, layers, step):
                qs.qs_sim_apply_layers_dev(sim.sim, dev[shift].data_ptr() + 4 * shift, c.layer_ptr, l, l + step)
            out.append(qs.qs_sim_tableau_export(sim.sim))
            sim.measure(np.arange(n, dtype=np.uint32), 1)
            out.append(sim.sample(70, 3, on_device=False))
            sim.sync()
        for i in (2, 4):
            assert np.array_equal(out[0], out[i]) and np.array_equal(out[1], out[i + 1]), (n, layers)
