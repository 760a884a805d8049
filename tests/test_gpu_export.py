"""The packed rows exported to host and device memory: small tableaus in one kernel, larger ones by copies, signs that
do not start on a word boundary."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 127, 500, 720, 760, 3_000])
def test_host_and_device_exports_agree_with_single_rows(n):
    import torch
    sim = qs.Simulator(n)
    sim.run(C.gate_mix_circuit(n, 10, seed=n, measure_every=5, measure_frac=0.3), seed=2)
    host = qs.qs_sim_tableau_export(sim.sim)
    k, words = (n + 63) // 64, len(host)
    dev = torch.full((words + 1,), 7, dtype=torch.int64, device="cuda")
    qs.qs_sim_tableau_export(sim.sim, out=dev)
    assert np.array_equal(dev.cpu().numpy().view(np.uint64)[:words], host) and int(dev[-1]) == 7
    x, z, r = sim.export_rows(np.arange(2 * n, dtype=np.uint32))
    rows = np.ascontiguousarray(host[:4 * n * k].reshape(2 * n, 2, k))
    bits = np.unpackbits(rows.view(np.uint8), axis=2, bitorder="little")
    assert np.array_equal(bits[:, 0, :n], x) and np.array_equal(bits[:, 1, :n], z)
    signs = np.unpackbits(np.ascontiguousarray(host[4 * n * k:]).view(np.uint8), bitorder="little")
    assert np.array_equal(signs[:2 * n], r) and not signs[2 * n:].any()
    assert not bits[:, :, n:].any()
