"""Batch circuits in shared memory: rounds of 7, 8, 9 and 17 measurements (passes of eight) with repeated
qubits, and their frame samples, equal to a simulator of the circuit alone."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


def _circuit(n):
    c = C.gate_mix_circuit(n, 10, seed=n, final_measure_all=False)
    rng = np.random.default_rng(n)
    c.ops = []
    for i, m in enumerate((7, 8, 9, 17, 1)):
        q = rng.integers(0, n, m).astype(np.uint32)
        q[-1] = q[0]
        c.ops += [("layers", 2 * i, 2 * i + 2), ("measure", q)]
    return c


def test_passes_of_eight_and_samples_equal_a_simulator():
    sizes = [1, 2, 64, 65, 127, 129, 256, 257, 448, 512, 640, 700, 900]
    circs = [_circuit(n) for n in sizes]
    shots = [1, 64, 65, 130, 300, 200, 256, 257, 100, 513, 129, 128, 192]
    b = qs.Batch(circs, list(range(len(sizes))))
    b.run()
    words = b.sample(shots, [7 + i for i in range(len(sizes))])
    b.sync()
    for i, c in enumerate(circs):
        s = qs.Simulator(c.n)
        assert np.array_equal(b.record(i), s.run(c, seed=i)), c.n
        rows = np.arange(2 * c.n, dtype=np.uint32)
        for u, v in zip(b.export_rows(i, rows), s.export_rows(rows)):
            assert np.array_equal(u, v), c.n
        want = s.sample(shots[i], 7 + i, on_device=False)
        assert np.array_equal(words[i].cpu().numpy().view(np.uint64), want), c.n


def test_records_follow_the_last_run():
    """Records after a partial run, a whole one and a partial one again; a count beyond what a
    simulator's circuit has measured is refused."""
    sizes = [50, 640, 700, 1_100]
    circs = [_circuit(n) for n in sizes]
    b = qs.Batch(circs, [1, 2, 3, 4])
    want = [qs.Simulator(c.n).run(c, seed=i + 1) for i, c in enumerate(circs)]
    lib, ptr = qs.lib(), qs.ctypes.c_void_p
    for limit, m in ((2, 15), (0, 42), (1, 7)):
        b.run(None, round_limit=limit)
        for i in range(len(sizes)):
            out = np.full(m, 9, np.uint8)
            assert lib.qs_batch_record(ptr(b.h), i, out.ctypes.data, m) == 0
            assert np.array_equal(out, want[i][:m]), (limit, sizes[i])
        out = np.zeros(42, np.uint8)
        assert (lib.qs_batch_record(ptr(b.h), 3, out.ctypes.data, 42) == 0) == (limit == 0)
