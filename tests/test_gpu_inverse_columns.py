"""Inverse-tableau measurement by columns: register widths of the kernels (32 W
words per column half), blocks of 64 or 32 with a partial last one, qubits
repeated inside a block and across blocks, and a qubit out of range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O  # noqa: E402
from paper_2603_14641_gb300 import qs  # noqa: E402
from workloads import circuits as C  # noqa: E402

INV = qs.QS_FLAG_INVERSE_TABLEAU


def _window(n, count, seed):
    rng = np.random.default_rng(seed)
    q = rng.integers(0, n, count).astype(np.uint32)
    q[count // 2:count // 2 + 5] = q[:5]  # repeats: inside a block, or in a later one
    return q


@pytest.mark.parametrize("n,count", [(1, 3), (33, 65), (128, 64), (129, 127), (512, 130), (1024, 63), (1025, 129)])
def test_windows_equal_the_inverse_oracle(n, count):
    circ = C.gate_mix_circuit(n, 12, seed=n, final_measure_all=False)
    sim = qs.Simulator(n, device="cuda:0", flags=INV)
    sim.run(circ, seed=0)
    inv, _, _ = O.run_circuit_inverse(circ, seed=0)
    m = 0
    for part, seed in ((count, 1), (1, 2), (count, 3)):
        q = _window(n, part, seed + n) if part > 10 else np.array([n - 1] * part, np.uint32)
        out = sim.measure(q, seed=7, shot=4)
        oout, kinds = inv.measure(q, seed=7, shot=4)
        assert np.array_equal(out, oout)
        assert np.array_equal(sim.record_kinds()[m:m + len(q)], kinds)
        m += len(q)
    x, z, _ = sim.export()
    ox, oz, oss, osd = inv.get()
    ss, sd = sim.qubit_signs()
    assert np.array_equal(x, ox) and np.array_equal(z, oz)
    assert np.array_equal(ss, oss) and np.array_equal(sd, osd)


@pytest.mark.parametrize("n", [2048, 2049, 4096, 4097, 8192, 8193, 16_384, 16_385])
def test_records_equal_the_chp_path_through_later_layers(n):
    circ = C.random_circuit(n, 8, 0.5, seed=n, final_measure_all=False)
    windows = [_window(n, 150, n + i) for i in range(3)]
    outs = []
    for flags in (INV, 0):
        s = qs.Simulator(n, device="cuda:0", flags=flags)
        dc = s.upload(circ)
        rec = []
        for q in windows:  # layers between the windows carry bits and signs on
            s.apply_layers_dev(dc, 0, circ.n_layers)
            rec.append(s.measure(q, seed=3))
        outs.append((np.concatenate(rec), s.record_kinds()))
        s.sync()
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])


def test_a_qubit_out_of_range_is_flagged_and_skipped():
    n = 100
    sim = qs.Simulator(n, device="cuda:0", flags=INV)
    sim.measure_dev(torch.tensor([5, n, 9], dtype=torch.int32, device="cuda:0"), seed=1)
    with pytest.raises(qs.QsError):
        sim.sync()
