"""Depolarising noise where blocks change between dealing the fired shots over their threads and drawing each
item's own (16 fired shots an item: p = 0.25), full and partial blocks of 256 items."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [0.2, 0.25, 0.3, 0.9, 1.0])
@pytest.mark.parametrize("kind", [C.DEPOLARIZE1, C.DEPOLARIZE2])
def test_fired_shots_around_the_switch(kind, p):
    n, shots = 54, 64 * 29 + 3
    c = C.random_circuit(n, 2, 0.5, seed=7)
    ops = [("layers", 0, 1), ("noise", kind, p, np.arange(n, dtype=np.uint32)), ("layers", 1, 2), c.ops[-1]]
    c = C.Circuit(n=n, gates=c.gates, layer_ptr=c.layer_ptr, ops=ops)
    sim = qs.Simulator(n)
    rec = sim.run(c, seed=4)
    bits = np.unpackbits(sim.sample(shots, seed=8, on_device=False).view(np.uint8), axis=1, bitorder="little")
    assert np.array_equal(bits[:, :shots], O.frames(c, rec, shots, seed=8))
