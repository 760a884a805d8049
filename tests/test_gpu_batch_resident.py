"""The batch's default path, a block per circuit of up to 640 qubits, at the edges of its size classes
(256 / 257, 448 / 449, 640 / 641 qubits) and of its 64-qubit blocks."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 63, 64, 65, 128, 256, 257, 448, 449, 640, 641, 700]


def _program(n, seed):
    """Gates of the whole set; rounds with repeated qubits (deterministic outcomes), one of them of
    more than 1,024 measurements, one empty, and one without gates before it."""
    c = C.gate_mix_circuit(n, 9, seed=seed, final_measure_all=False)
    rng = np.random.default_rng(seed)

    def some(m):
        return ("measure", rng.integers(0, n, m).astype(np.uint32))

    c.ops = [("layers", 0, 4), some(min(n, 40)), some(5), ("layers", 4, 5), ("measure", np.zeros(0, np.uint32)),
             ("layers", 5, 8), some(1100 if n <= 128 else 70), ("layers", 8, 9)]
    return c


def test_resident_batch_matches_oracle_and_simulator():
    circs = [_program(n, 50 + n) for n in SIZES]
    seeds = [3 * n + 1 for n in SIZES]
    b = qs.Batch(circs, seeds, shot=2)
    for _ in range(2):  # the second run starts from |0...0> again
        b.run()
        b.sync()
    for i, c in enumerate(circs):
        rows = np.arange(2 * c.n, dtype=np.uint32)
        got = b.export_rows(i, rows)
        if c.n <= 260:
            o, rec, _ = O.run_circuit(c, seed=seeds[i], shot=2)
            want = o.get()
        else:
            s = qs.Simulator(c.n)
            rec = s.run(c, seed=seeds[i], shot=2)
            want = s.export_rows(rows)
        assert np.array_equal(b.record(i), rec), c.n
        for u, v in zip(got, want):
            assert np.array_equal(u, v), c.n


def test_round_limit_and_launch_shape_agree():
    """The first rounds only, on the default path and on the persistent kernel, then a whole run."""
    circs = [C.random_circuit(n, 12, 0.5, seed=n, measure_every=3, measure_frac=0.2, final_measure_all=False)
             for n in (40, 300, 650, 1100)]
    b = qs.Batch(circs, [5, 6, 7, 8])
    out = []
    for tuning in (None, qs.qs_batch_tuning(512, 0, 1, 0, 0), qs.qs_batch_tuning(0, 0, 0, 0, 0)):
        b.run(tuning, round_limit=2)
        b.sync()
        part = [b.export_rows(i, np.arange(2 * c.n, dtype=np.uint32)) for i, c in enumerate(circs)]
        b.run(tuning)
        samples = [s.cpu().numpy() for s in b.sample([130] * 4, [1, 2, 3, 4])]
        b.sync()
        out.append((part, [b.record(i) for i in range(4)], samples))
    for other in out[1:]:
        for p, q in zip(out[0][0], other[0]):
            for u, v in zip(p, q):
                assert np.array_equal(u, v)
        for u, v in zip(out[0][1] + out[0][2], other[1] + other[2]):
            assert np.array_equal(u, v)
