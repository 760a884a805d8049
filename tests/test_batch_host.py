"""Host code of the batches on a CUDA runtime without a GPU: the autotuner's cache, the
launch shapes that are refused, and what creating a batch and reading its records costs."""
import ctypes

import numpy as np

from paper_2603_14641_gb300 import qs
from tests import fake_cuda
from workloads import circuits as C


def _create(circs):
    keep, arr = [], (qs.qs_batch_circuit * len(circs))()
    for i, c in enumerate(circs):
        g, lp = np.ascontiguousarray(c.gates, np.uint32), np.ascontiguousarray(c.layer_ptr, np.int64)
        rl, rm, q = qs.circuit_rounds(c)
        keep += [g, lp, rl, rm, q]
        arr[i] = qs.qs_batch_circuit(c.n, c.n_layers, g.ctypes.data, lp.ctypes.data, len(rl) - 1, 0, rl.ctypes.data,
                                     rm.ctypes.data, q.ctypes.data if q.size else None, i, 0)
    h = ctypes.c_void_p()
    assert qs.lib().qs_batch_create(len(circs), ctypes.byref(arr), None, None, 0, ctypes.byref(h)) == 0
    return h


def _circuits(sizes, depth=20, every=5):
    return [C.random_circuit(n, depth, 0.5, seed=n, measure_every=every, measure_frac=0.2, final_measure_all=False)
            for n in sizes]


def test_autotune_takes_no_line_of_another_choice(monkeypatch, tmp_path):
    """A line whose key lacks the set of candidates (the shapes of the persistent kernel alone) is not an answer."""
    L = fake_cuda.use(monkeypatch)
    circs = _circuits([50, 300, 900])
    h = _create(circs)
    sig, m64 = 1469598103934665603, (1 << 64) - 1
    for v in [len(circs)] + [x for c in circs for x in (c.n, len(qs.circuit_rounds(c)[0]) - 1, len(c.gates), c.n_measurements)]:
        sig = (sig ^ v) * 1099511628211 & m64
    path = tmp_path / "tune.txt"
    path.write_text(f"fake|{sig:016x}|0 512 1 1 0\n")
    t = qs.qs_batch_tuning()
    assert L.qs_batch_autotune(h, 0, str(path).encode(), ctypes.byref(t)) == 0
    assert t.threads == 0  # every candidate takes the same time here: the first is kept
    lines = path.read_text().splitlines()
    assert len(lines) == 2
    path.write_text(lines[1].split()[0] + " 256 2 1 1\n")  # a line of this choice is
    assert L.qs_batch_autotune(h, 0, str(path).encode(), ctypes.byref(t)) == 0
    assert (t.threads, t.blocks_per_sm, t.words_per_block, t.fuse_depth) == (256, 2, 1, 1)
    L.qs_batch_destroy(h)


def test_incomplete_launch_shapes_are_refused(monkeypatch):
    """threads = 0 asks for the default path only where nothing else of a launch shape is given. A batch
    without circuits for the persistent kernel does not look at the shape."""
    L = fake_cuda.use(monkeypatch)
    for sizes in ([50, 300], [1_024, 1_100]):
        h = _create(_circuits(sizes))
        for shape, ok in (((0, 0, 0, 0, 0), True), ((0, 0, 1, 0, 0), False), ((0, 2, 0, 0, 0), False),
                          ((0, 0, 0, 1, 0), False), ((0, 0, 0, 0, 9), True), ((512, 1, 1, 0, 0), True),
                          ((128, 1, 1, 0, 0), False)):
            rc = L.qs_batch_run(h, ctypes.byref(qs.qs_batch_tuning(*shape)), 0)
            assert rc == (0 if ok or sizes[0] > 1_000 else -1), (sizes, shape)
        L.qs_batch_destroy(h)


def test_create_uploads_a_circuit_in_three_copies(monkeypatch):
    """Gates, offsets and qubits; nothing is pinned, and all records come to the host in one copy."""
    L = fake_cuda.use(monkeypatch)
    circs = _circuits([5, 64, 640, 300, 17, 2])
    h = _create(circs)
    assert fake_cuda.count("pinned") == 0
    assert fake_cuda.count("copy") <= 3 * len(circs) + 4
    assert L.qs_batch_run(h, None, 0) == 0
    L.fake_reset(-1, 0)
    for i, c in enumerate(circs):
        out = np.zeros(max(c.n_measurements, 1), np.uint8)
        assert L.qs_batch_record(h, i, out.ctypes.data, c.n_measurements) == 0
    assert fake_cuda.count("copy") <= 2  # the error flags, the records
    L.qs_batch_destroy(h)


def test_simulators_of_a_batch_share_an_allocation(monkeypatch):
    """Circuits of 641 to 1,023 qubits run through simulators: one allocation for all, the batch's gate records."""
    L = fake_cuda.use(monkeypatch)
    circs = _circuits([700, 641, 1_023, 900, 800])
    h = _create(circs)
    assert fake_cuda.count("pinned") == 0
    assert fake_cuda.count("cudaMalloc") == 2  # the batch's workspace, the simulators
    assert fake_cuda.count("copy") <= 3 * len(circs) + 4
    assert L.qs_batch_run(h, None, 0) == 0
    L.qs_batch_destroy(h)


def test_sync_reads_the_flags_of_simulators_with_work(monkeypatch):
    """After a run those of every simulator, after sampling those of the circuits that sample through theirs."""
    L = fake_cuda.use(monkeypatch)
    circs = _circuits([700, 641, 1_023, 1_024, 1_100, 50])
    h = _create(circs)
    k, ow = len(circs), 2
    out = [np.zeros((c.n_measurements, ow), np.uint64) for c in circs]
    ptrs = (ctypes.c_void_p * k)(*[o.ctypes.data for o in out])
    shots, seeds = np.full(k, 128, np.uint64), np.zeros(k, np.uint64)
    for want, call in ((1 + 5, lambda: L.qs_batch_run(h, None, 0)),
                       (1 + 2, lambda: L.qs_batch_sample(h, shots.ctypes.data, seeds.ctypes.data,
                                                         ctypes.cast(ptrs, ctypes.c_void_p))),
                       (0, lambda: 0)):
        assert call() == 0
        L.fake_reset(-1, 0)
        assert L.qs_batch_sync(h) == 0
        assert fake_cuda.count("copy") == want
    L.qs_batch_destroy(h)


def test_a_run_that_stops_within_a_large_circuit_is_not_complete(monkeypatch):
    """Sampling needs the records of a complete run of every circuit, the large ones included."""
    L = fake_cuda.use(monkeypatch)
    circs = _circuits([50], every=10) + _circuits([1_100], every=2)
    assert [len(qs.circuit_rounds(c)[0]) - 1 for c in circs] == [2, 10]
    h = _create(circs)
    out = [np.zeros((c.n_measurements, 1), np.uint64) for c in circs]
    ptrs = (ctypes.c_void_p * 2)(*[o.ctypes.data for o in out])
    shots, seeds = np.full(2, 10, np.uint64), np.zeros(2, np.uint64)
    for limit, rc in ((3, -6), (9, -6), (10, 0), (0, 0)):
        assert L.qs_batch_run(h, None, limit) == 0
        got = L.qs_batch_sample(h, shots.ctypes.data, seeds.ctypes.data, ctypes.cast(ptrs, ctypes.c_void_p))
        assert got == rc, limit
    L.qs_batch_destroy(h)
