"""The first staged call of a simulator inside a stream capture: its pinned slot is allocated there, and the captured
copy carries the call's records."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2603_14641_gb300 import qs  # noqa: E402
from workloads import circuits as C  # noqa: E402


@pytest.mark.parametrize("n,flags", [(200, qs.QS_FLAG_INVERSE_TABLEAU), (17_000, 0)])
def test_host_layers_in_a_capture(n, flags):
    c = C.gate_mix_circuit(n, 3, seed=4, final_measure_all=False)
    plain = qs.Simulator(n, flags=flags)
    for l in range(3):
        plain.apply_layer(c.layer(l))
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        sim = qs.Simulator(n, flags=flags, stream=stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for l in range(3):
            sim.apply_layer(c.layer(l))
    graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(sim.export(), plain.export()):
        assert np.array_equal(a, b)
    sim.sync()
