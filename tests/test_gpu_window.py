"""Measurement windows with deterministic outcomes in them: they are evaluated together after the
window's last block, and the symbolic pass looks past the rows it holds when those have no pivot."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_14641_gb300 import qs
from workloads import circuits as C

pytestmark = pytest.mark.gpu


def _check(sim, o, rec, orec, okinds):
    assert np.array_equal(rec, orec)
    assert np.array_equal(sim.record_kinds(), okinds)
    for a, b in zip(sim.export(), o.get()):
        assert np.array_equal(a, b)
    sim.sync()


# 2,100 qubits: two 32-word column chunks. depth 2: sparse columns, most outcomes of the second pass
# deterministic. 2,600 dense qubits with repeats: more than 1,024 nonzero rows and steps without a
# pivot among them, so the symbolic pass scans the rest. One repeat only: the rows of its product are
# split over blocks. 97 repeats: several groups of 32, the last one short.
@pytest.mark.parametrize("flags", [0, qs.QS_FLAG_STEP_SYMBOLIC])
@pytest.mark.parametrize("n,depth,first,again", [(70, 3, 70, 33), (300, 2, 150, 97), (2100, 2, 130, 97),
                                                 (2600, 60, 40, 1), (2600, 60, 40, 97), (1030, 40, 64, 64)])
def test_window_with_deterministic_outcomes(n, depth, first, again, flags):
    circ = C.random_circuit(n, depth, 0.5, seed=n + depth, final_measure_all=False)
    rng = np.random.default_rng(n + again)
    q = rng.permutation(n)[:first].astype(np.uint32)
    # repeats of measured qubits between and after the first measurements of others
    q = np.concatenate([q[:first // 2], rng.choice(q[:first // 2], again // 2), q[first // 2:],
                        rng.choice(q, again - again // 2)]).astype(np.uint32)
    sim = qs.Simulator(n, flags=flags)
    dc = sim.upload(circ)
    sim.apply_layers_dev(dc, 0, depth)
    rec = sim.measure(q, seed=5, shot=3)
    o = O.Oracle(n)
    o.apply(circ.gates)
    orec, okinds = o.measure(q, seed=5, shot=3)
    _check(sim, o, rec, orec, okinds)


def test_out_of_range_device_qubit_in_a_window():
    """A device list is not checked on the host: the outcome is 0 and the next sync reports it."""
    import torch
    sim = qs.Simulator(100)
    q = np.arange(40, dtype=np.int32)
    q[7] = 100
    dev = torch.from_numpy(q).cuda()
    sim.measure_dev(dev, seed=1)
    with pytest.raises(qs.QsError) as e:
        sim.sync()
    assert e.value.code == -7


# 255..257 and 511..513: 4- and 8-word chunks of the small apply pass (row strides 4, 8 and 12 words,
# the last with a half-empty chunk); 6,144 / 6,145: the last small and the first large size
@pytest.mark.parametrize("n,flags", [(255, 0), (257, 0), (512, 0), (513, 0), (6144, 0), (6145, 0),
                                     (6145, qs.QS_FLAG_WIDE_OFFSETS)])
def test_apply_variants_match_single_measurements(n, flags):
    """Blocks of 64 (the second one short) against measurements one by one, on a dense state."""
    circ = C.random_circuit(n, 30, 0.5, seed=n, final_measure_all=False)
    q = np.random.default_rng(n).permutation(n)[:100].astype(np.uint32)
    out = []
    for f in (flags, qs.QS_FLAG_NO_BLOCKED_MEASURE):
        sim = qs.Simulator(n, flags=f)
        dc = sim.upload(circ)
        sim.apply_layers_dev(dc, 0, 30)
        rec = sim.measure(q, seed=2)
        out.append((rec, sim.record_kinds(), qs.qs_sim_tableau_export(sim.sim)))
        sim.sync()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n,layers", [(1, 3), (5, 2), (64, 9), (130, 7), (700, 6), (14081, 5)])
def test_deferred_gates_match_layer_by_layer(n, layers):
    """A run of layers defers its one-qubit gates to the next two-qubit gate of their qubit; one layer
    per call applies each in its own layer. All 11 gates, an empty layer and a layer of identities."""
    c = C.gate_mix_circuit(n, layers, seed=n, final_measure_all=False)
    ident = np.array([[C.I, q, 0] for q in range(min(n, 3))], np.uint32)
    lp = c.layer_ptr
    gates = np.concatenate([c.gates[:lp[1]], ident, c.gates[lp[1]:]])
    lp = np.concatenate([lp[:2], lp[1:2], [lp[1] + len(ident)], lp[2:] + len(ident)])
    c = C.Circuit(n=n, gates=np.ascontiguousarray(gates), layer_ptr=lp, ops=[])
    out = []
    for together in (True, False):
        sim = qs.Simulator(n, flags=qs.QS_FLAG_NO_FUSION)
        sim.reset(np.arange(n) % 3 == 1)
        dc = sim.upload(c)
        for l in range(1 if together else c.n_layers):
            sim.apply_layers_dev(dc, l, c.n_layers if together else l + 1)
        out.append(qs.qs_sim_tableau_export(sim.sim))
        sim.sync()
    assert np.array_equal(*out)
    if n <= 130:
        o = O.Oracle(n, (np.arange(n) % 3 == 1).astype(np.uint8))
        o.apply(c.gates)
        assert all(np.array_equal(a, b) for a, b in zip(qs.unpack_rows(out[0], n), o.get()))
