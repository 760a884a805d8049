"""Host layers whose records go with the launch: equal to the same layers from
device memory at the edges of the record counts and of the qubit numbers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_14641_gb300 import qs  # noqa: E402


def _layer(n, n_gates, seed):
    """n_gates gates of all types on distinct qubits, the highest qubit included."""
    rng = np.random.default_rng(seed)
    perm = rng.permutation(n - 1)
    pool = np.concatenate([[n - 1], perm])
    two = min(n_gates, n - n_gates)
    g = np.zeros((n_gates, 3), np.uint32)
    g[:, 0] = rng.integers(0, 7, n_gates)  # I .. SDG
    g[:, 1] = pool[:n_gates]
    g[:two, 0] = 7 + np.arange(two) % 5  # CX .. ISWAP
    g[:two, 2] = pool[n_gates:n_gates + two]
    return g[rng.permutation(n_gates)]


@pytest.mark.parametrize("n,n_gates", [(1, 1), (2, 1), (129, 127), (200, 128), (200, 129), (1000, 512), (1000, 513),
                                       (3000, 2048), (3000, 2049), (16_384, 2048), (16_385, 300)])
def test_host_layers_equal_device_layers(n, n_gates):
    layers = [_layer(n, n_gates, i) for i in range(3)]
    a, b = qs.Simulator(n), qs.Simulator(n)
    ptr = np.arange(4, dtype=np.int64) * n_gates
    packed = torch.from_numpy(qs.qs_pack_layers(n, np.concatenate(layers), ptr).view(np.int32)).cuda()
    for i, g in enumerate(layers):
        a.apply_layer(g)
        qs.qs_sim_apply_layers_dev(b.sim, packed.data_ptr(), ptr, i, i + 1)
    for u, v in zip(a.export(), b.export()):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("n,flags", [(300, qs.QS_FLAG_NO_FUSION), (15_000, 0)])
def test_unfused_device_records_need_four_byte_alignment_only(n, flags):
    layers = [_layer(n, n // 2, i) for i in range(5)]
    ptr = np.arange(6, dtype=np.int64) * (n // 2)
    packed = qs.qs_pack_layers(n, np.concatenate(layers), ptr).view(np.int32)
    out = []
    for shift in (0, 1):
        dev = torch.zeros(len(packed) + 1, dtype=torch.int32, device="cuda")
        dev[shift:shift + len(packed)] = torch.from_numpy(packed).cuda()
        sim = qs.Simulator(n, flags=flags)
        qs.qs_sim_apply_layers_dev(sim.sim, dev.data_ptr() + 4 * shift, ptr, 0, 5)
        out.append(qs.qs_sim_tableau_export(sim.sim))
        sim.sync()
    assert np.array_equal(*out)
