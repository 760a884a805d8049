"""Chained measurement launches (a kernel may be resident before the one ahead of it ends): many blocks of 64 one
after the other, several times over and on several streams at once, equal to measuring one by one."""
import numpy as np
import pytest

from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,flags", [((300, 1_500, 700), 0), ((6_144, 7_000, 200), 0),
                                         ((500, 2_000, 1_030), qs.QS_FLAG_INVERSE_TABLEAU)])
def test_blocks_in_flight_on_several_streams(sizes, flags):
    import torch
    sims = []
    for n in sizes:
        c = C.random_circuit(n, 8, 0.5, seed=n, measure_every=4, measure_frac=0.05)
        ref = qs.Simulator(n, flags=qs.QS_FLAG_NO_BLOCKED_MEASURE)
        want = ref.run(c, seed=5)
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            sim = qs.Simulator(n, flags=flags)
            sims.append((sim, c, sim.upload(c), want))
    torch.cuda.synchronize()
    for _ in range(4):
        for sim, c, dc, _w in sims:
            sim.reset()
            for op in c.ops:
                if op[0] == "layers":
                    sim.apply_layers_dev(dc, op[1], op[2])
                else:
                    sim.measure(op[1], seed=5, want_outcomes=False)
        for sim, _c, _d, want in sims:
            assert np.array_equal(sim.record(), want)
            sim.sync()
