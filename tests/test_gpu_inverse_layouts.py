"""Inverse mode: calls of one or a few measurements go by rows where the whole tableau by columns costs more,
larger ones by columns; bits, signs and records are the same whichever way each call goes."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from tests import fake_cuda
from workloads import circuits as C

INV = qs.QS_FLAG_INVERSE_TABLEAU


@pytest.mark.gpu
@pytest.mark.parametrize("n", [7_000, 9_000])
def test_mixed_calls_equal_one_window(n):
    c = C.random_circuit(n, 8, 0.5, seed=n, final_measure_all=False)
    q = np.random.default_rng(n).integers(0, n, 60).astype(np.uint32)
    q[40:45] = q[:5]
    out = []
    for cuts in ([60], [1, 1, 40, 1, 2, 15], [1] * 60):
        sim = qs.Simulator(n, flags=INV)
        dc = sim.upload(c)
        for _ in range(2):
            sim.apply_layers_dev(dc, 0, 8)
            at = 0
            for m in cuts:
                sim.measure(q[at:at + m], seed=3)
                at += m
        out.append([sim.record(), sim.record_kinds(), qs.qs_sim_tableau_export(sim.sim), *sim.qubit_signs()])
        sim.sync()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n,few,many", [(2_000, 0, 1), (9_000, 2, 3), (16_000, 5, 6), (16_385, 70, 0)])
def test_few_measurements_take_rows(monkeypatch, n, few, many):
    """With both layouts at hand: four launches a measurement against two a block."""
    fake_cuda.use(monkeypatch)
    s = qs.qs_sim_create(n, flags=INV)
    for count in ([few] if few else []) + ([many] if many else []):
        qs.qs_sim_reset(s)
        qs.qs_sim_tableau_export(s, out=np.zeros(2 * n * 2 * ((n + 63) // 64) + (2 * n + 63) // 64, np.uint64))
        before = fake_cuda.count("launch")
        qs.qs_sim_measure(s, np.arange(count), 1)
        launches = fake_cuda.count("launch") - before
        assert launches == (1 + 4 * count if count == few else 3), (count, launches)
    qs.qs_sim_destroy(s)
