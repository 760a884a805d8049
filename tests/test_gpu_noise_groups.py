"""Noise ops that launch together (consecutive, distinct qubits, four at most) and those that must not,
with items (targets x 64-shot words) around a block's 256."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shots", [1, 64, 65, 640, 8_200])
@pytest.mark.parametrize("p", [0.004, 0.6, 1.0])
def test_runs_of_noise_ops_match_oracle(shots, p):
    n = 60
    c = C.random_circuit(n, 4, 0.5, seed=3)
    q = np.random.default_rng(5).permutation(n).astype(np.uint32)
    noise = [("noise", C.NOISE_X, p, q[:13]), ("noise", C.DEPOLARIZE2, p, q[13:39]), ("noise", C.NOISE_Z, 0.0, q[39:41]),
             ("noise", C.DEPOLARIZE1, p, q[41:]),                    # four on distinct qubits
             ("noise", C.NOISE_Y, p, q[:1]),                         # a fifth: starts a new run
             ("noise", C.DEPOLARIZE1, p, q[:1]),                     # same qubit again: another run
             ("noise", C.DEPOLARIZE2, p, q[:40]), ("noise", C.DEPOLARIZE2, p, q[40:])]
    ops = [("layers", 0, 2)] + noise + [("layers", 2, 4)] + noise[3:] + [("measure", np.arange(n, dtype=np.uint32))]
    c = C.Circuit(n=n, gates=c.gates, layer_ptr=c.layer_ptr, ops=ops)
    sim = qs.Simulator(n)
    rec = sim.run(c, seed=4)
    words = sim.sample(shots, seed=8, on_device=False)
    bits = np.unpackbits(words.view(np.uint8), axis=1, bitorder="little")
    assert not bits[:, shots:].any()
    assert np.array_equal(bits[:, :shots], O.frames(c, rec, shots, seed=8))
