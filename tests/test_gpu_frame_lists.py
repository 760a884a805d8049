"""Sampled windows of every way a qubit list reaches the kernel: 128 and 1,024 in a launch's parameters, two
launches, and beyond that through the device, equal to windows of one measurement each."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,count", [(1, 1), (200, 128), (200, 129), (1_100, 1_024), (1_100, 1_025), (2_100, 2_048),
                                     (2_100, 2_049)])
def test_windows_of_any_length_sample_the_same(n, count):
    c = C.random_circuit(n, 6, 0.5, seed=n, final_measure_all=False)
    q = np.random.default_rng(n).permutation(n)[:count].astype(np.uint32)
    out = []
    for split in (False, True):
        sim = qs.Simulator(n)
        sim.apply_layers_dev(sim.upload(c), 0, 6)
        for part in (np.array_split(q, 13) if split and count > 13 else [q]):
            sim.measure(part, seed=4, want_outcomes=False)
        out.append(sim.sample(130, seed=9, on_device=False))
        if n <= 200:
            words = np.zeros((count, 3), np.uint64)
            qs.qs_sim_sample_noalloc(sim.sim, 130, 9, words.ctypes.data, words.size)
            out.append(words)
        sim.sync()
    for o in out[1:]:
        assert np.array_equal(np.asarray(o).view(np.uint64), out[0])


@pytest.mark.parametrize("count", [1, 255, 256, 257, 2_048, 2_049])
def test_host_lists_equal_device_lists(count):
    import torch
    n = 2_100
    c = C.random_circuit(n, 6, 0.5, seed=n, final_measure_all=False)
    q = np.random.default_rng(count).integers(0, n, count).astype(np.uint32)
    a, b = qs.Simulator(n), qs.Simulator(n)
    for s in (a, b):
        s.apply_layers_dev(s.upload(c), 0, 6)
    got = a.measure(q, seed=4)
    b.measure_dev(torch.from_numpy(q.view(np.int32)).cuda(), seed=4)
    assert np.array_equal(got, b.record())
    for u, v in zip(a.export(), b.export()):
        assert np.array_equal(u, v)
