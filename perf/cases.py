"""What users of the simulator run, as measurable cases.

Every case is one call sequence of the public Python API (qs.Simulator, qs.Batch), which only
marshals arguments for the C ABI. A case is a dict of plain values; "kind" says what is called:

  job      a circuit resident in device memory, from |0...0>: layers, Z-measurements (a share of the
           qubits every `every` layers, then `final` qubits, all if 0) and frame samples. Returns the
           outcomes of the record and the samples, and with "state" the tableau the program goes on with
           (packed rows, in device memory).
  host     the simplest use: every layer and the measured qubits come from host arrays, outcomes and
           the whole tableau go back to the host. Gates from the whole 11-gate set.
  evolve   gate layers alone; returns the tableau in the device's own layout, in device memory.
  remeasure a shallow circuit and `rounds` rounds of measurements of every qubit: a mixture of
           probabilistic and deterministic outcomes, then deterministic ones only. Returns the
           outcomes, their kinds and the tableau (packed rows, in device memory).
  sample   many shots of a program that has run (its reference record is there), noiseless or with
           circuit-level Pauli noise.
  batch    independent circuits as one qs.Batch: run, then sample every circuit.

Inputs (random Clifford circuits of workloads/circuits.py) come from the seed alone. Every result is
a bit or a word of bits: all of them have to be equal, and there is no rounding.
"""
import math
import random

import numpy as np
import torch

from paper_2603_14641_gb300 import qs
from workloads import circuits as W

MAX_BATCH = 56  # circuits of one batch case: each returns its own samples


def listed():
    return [
        # the 256-qubit workload (depth 100, every qubit measured at the end): one small program, where
        # launches and waits count
        dict(name="job_n256", kind="job", n=256, depth=100, p_cx=0.5, every=0, frac=0.0, final=0, shots=1024, state=False, inverse=False),
        # a first user's program through host arrays, at the small end of the paper's qubit range (100)
        dict(name="host_n127", kind="host", n=127, depth=60),
        # the 10,000-qubit workload in full: 1,000 layers, 5% of the qubits measured every 50 layers and
        # all at the end (19,500 measurements)
        dict(name="job_n10000", kind="job", n=10_000, depth=1_000, p_cx=0.5, every=50, frac=0.05, final=0, shots=1024, state=True, inverse=False),
        # the 180,000-qubit workload with its first 100 layers (the paper's smallest depth; the state is
        # dense by then), a part of its final measurement and samples: every tableau pass runs at HBM size
        dict(name="job_n180000", kind="job", n=180_000, depth=100, p_cx=0.4, every=0, frac=0.0, final=2_048, shots=1024, state=False, inverse=False),
        # the same generator at its 20,000-qubit size, every qubit measured: the measurement-bound job
        dict(name="job_n20000", kind="job", n=20_000, depth=100, p_cx=0.4, every=0, frac=0.0, final=0, shots=256, state=True, inverse=False),
        # tableau evolution alone above the sizes that fit shared memory slices, a ragged size
        dict(name="evolve_n30001", kind="evolve", n=30_001, depth=60, p_cx=0.4),
        # readout of a shallow circuit, twice (the second round repeats the first one's outcomes)
        dict(name="remeasure_n1500", kind="remeasure", n=1_500, depth=3, p_cx=0.5, rounds=2),
        # a served request's shots (the serving mix: 100..20,000 qubits, 1e3..1e6 shots)
        dict(name="sample_n1000", kind="sample", n=1_000, depth=200, shots=200_000, p=0.0),
        # noisy shots: depolarising noise after every layer, flips before the readout
        dict(name="sample_noisy_n4999", kind="sample", n=4_999, depth=50, shots=16_384, p=1e-3),
        # the batched workload (n log-uniform 50..5,000, 10% of the qubits measured every 10 layers)
        dict(name="batch_mixed", kind="batch", count=40, lo=50, hi=5_000, depth=100, shots=256),
        # small requests that a server runs together as one batch
        dict(name="batch_small", kind="batch", count=56, lo=50, hi=1_000, depth=100, shots=2_048),
        # the paper's own measurement variant (qubit-indexed signs of the inverse tableau)
        dict(name="inverse_n2000", kind="job", n=2_000, depth=100, p_cx=0.5, every=50, frac=0.05, final=0, shots=1024, state=False, inverse=True),
    ]


def _log(rng, lo, hi):
    """A whole number, log-uniform in [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["small", "mid", "large", "final", "host", "evolve", "remeasure", "sample", "noisy",
                       "batch", "inverse"])
    if kind == "host":
        return dict(kind="host", n=_log(rng, 20, 1_500), depth=rng.randint(10, 100))
    if kind == "evolve":
        return dict(kind="evolve", n=_log(rng, 500, 40_000), depth=rng.randint(10, 60), p_cx=round(rng.uniform(0.2, 0.8), 2))
    if kind == "remeasure":
        return dict(kind="remeasure", n=_log(rng, 200, 3_000), depth=rng.randint(1, 6), p_cx=round(rng.uniform(0.3, 0.7), 2),
                    rounds=rng.randint(1, 2))
    if kind == "sample":
        n = _log(rng, 100, 20_000)
        return dict(kind="sample", n=n, depth=rng.randint(20, 200), shots=_log(rng, 1_000, min(1_000_000, 400_000_000 // n)), p=0.0)
    if kind == "noisy":
        n = _log(rng, 100, 10_000)
        return dict(kind="sample", n=n, depth=rng.randint(10, 50), shots=_log(rng, 500, min(100_000, 80_000_000 // n)),
                    p=rng.choice([1e-4, 1e-3, 1e-2]))
    if kind == "batch":
        lo = rng.choice([50, 50, 200])
        return dict(kind="batch", count=rng.randint(8, MAX_BATCH), lo=lo, hi=_log(rng, 300, 5_000), depth=rng.randrange(20, 101, 10),
                    shots=_log(rng, 64, 4_096))
    if kind == "large":
        return dict(kind="job", n=_log(rng, 40_000, 170_000), depth=_log(rng, 5, 100), p_cx=round(rng.uniform(0.3, 0.6), 2), every=0,
                    frac=0.0, final=_log(rng, 64, 2_048), shots=_log(rng, 64, 1_024), state=False, inverse=False)
    if kind == "final":
        return dict(kind="job", n=_log(rng, 4_000, 20_000), depth=_log(rng, 5, 100), p_cx=round(rng.uniform(0.3, 0.6), 2), every=0,
                    frac=0.0, final=0, shots=_log(rng, 64, 1_024), state=True, inverse=False)
    every = rng.choice([0, 10, 25, 50])
    n = {"small": (64, 1_200), "mid": (1_200, 13_000), "inverse": (64, 2_500)}[kind]
    return dict(kind="job", n=_log(rng, *n), depth=rng.randint(50, 150), p_cx=round(rng.uniform(0.3, 0.6), 2), every=every,
                frac=0.05 if every else 0.0, final=0, shots=_log(rng, 64, 4_096), state=kind == "mid", inverse=kind == "inverse")


def _batch_circuits(case, seed):
    # sizes log-uniform in [lo, hi], the case's own: the seed draws the circuits
    r = np.random.Generator(np.random.PCG64(case["count"]))
    sizes = np.round(np.exp(r.uniform(np.log(case["lo"]), np.log(case["hi"]), size=case["count"]))).astype(int)
    return [W.random_circuit(int(n), case["depth"], 0.5, seed=seed * 1_009 + i, measure_every=10, measure_frac=0.1,
                             final_measure_all=False) for i, n in enumerate(sizes)]


def _circuit(case, seed):
    c = W.random_circuit(case["n"], case["depth"], case["p_cx"], seed=seed, measure_every=case["every"], measure_frac=case["frac"])
    if case["final"]:
        c.ops[-1] = ("measure", np.arange(case["final"], dtype=np.uint32))
    return c


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind == "batch":
        cs = _batch_circuits(case, seed)
        st["batch"] = qs.Batch(cs, [seed + i for i in range(len(cs))])
        return st
    n = case["n"]
    if kind == "host":
        c = W.gate_mix_circuit(n, case["depth"], seed)
    elif kind == "job":
        c = _circuit(case, seed)
    elif kind == "sample":
        c = W.random_circuit(n, case["depth"], 0.5, seed=seed)
        if case["p"]:
            c = W.with_circuit_noise(c, case["p"], case["p"])
    else:
        c = W.random_circuit(n, case["depth"], case["p_cx"], seed=seed)
    st["circuit"] = c
    st["sim"] = sim = qs.Simulator(n, flags=qs.QS_FLAG_INVERSE_TABLEAU if case.get("inverse") else 0)
    if kind != "host":
        st["dc"] = sim.upload(c)
    if kind == "sample":  # the program has run once: its record is the reference of the shots
        sim.run(c, seed, dc=st["dc"])
    k = (n + 63) // 64
    if kind == "evolve":
        st["out"] = torch.empty((2 * n + 1) * ((2 * k + 3) // 4 * 4), dtype=torch.int64, device="cuda")
    elif kind == "remeasure" or case.get("state"):
        st["out"] = torch.empty(2 * n * 2 * k + (2 * n + 63) // 64, dtype=torch.int64, device="cuda")
    return st


def run(st):
    case, kind, seed = st["case"], st["case"]["kind"], st["seed"]
    if kind == "batch":
        b = st["batch"]
        b.run()
        samples = b.sample([case["shots"]] * case["count"], [seed + 1 + i for i in range(case["count"])])
        b.sync()
        return np.concatenate([b.record(i) for i in range(case["count"])]), samples
    sim, c = st["sim"], st["circuit"]
    if kind == "sample":
        return sim.sample(case["shots"], seed + 1)
    sim.reset()
    if kind == "job":
        record = sim.run(c, seed, dc=st["dc"])
        samples = sim.sample(case["shots"], seed + 1)
        if case["state"]:
            return record, samples, qs.qs_sim_tableau_export(sim.sim, out=st["out"])
        return record, samples
    if kind == "host":
        for l in range(c.n_layers):
            sim.apply_layer(c.layer(l))
        outcomes = sim.measure(np.arange(case["n"], dtype=np.uint32), seed)
        return outcomes, qs.qs_sim_tableau_export(sim.sim)
    sim.apply_layers_dev(st["dc"], 0, c.n_layers)
    if kind == "evolve":
        return qs.qs_sim_tableau_export(sim.sim, qs.QS_LAYOUT_NATIVE, out=st["out"])
    q = np.arange(case["n"], dtype=np.uint32)
    rounds = [sim.measure(q, seed) for _ in range(case["rounds"])]
    return rounds, sim.record_kinds(), qs.qs_sim_tableau_export(sim.sim, out=st["out"])


def work(case):
    """Bytes: gate records (8 a gate, about 0.83 n gates a layer at p_cx 0.5), the tableau (n^2 / 2
    bytes) written once, and read and written once more where measurements change it, frames written
    and read once, outputs. Bit operations only: no floating-point work."""
    def one(n, depth, meas, shots, tableau=True):
        gates = 8.0 * 0.8 * n * depth
        frames = 2 * (2 * n * shots / 8) if shots else 0
        return gates + (n * n / 2) * ((1 + (2 if meas else 0)) if tableau else 0) + frames + meas * (1 + shots / 8)

    kind = case["kind"]
    if kind == "batch":
        n = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": case["count"] * one(n, case["depth"], 0.1 * n * case["depth"] / 10, case["shots"]), "flops": 0}
    n, depth = case["n"], case["depth"]
    if kind == "host":
        return {"bytes": one(n, depth, n, 0) + n * n / 2, "flops": 0}
    if kind == "evolve":
        return {"bytes": one(n, depth, 0, 0), "flops": 0}
    if kind == "remeasure":
        return {"bytes": one(n, depth, n * case["rounds"], 0), "flops": 0}
    if kind == "sample":
        return {"bytes": one(n, depth, n, case["shots"], tableau=False), "flops": 0}
    meas = (case["final"] or n) + (n * case["frac"] * (depth // case["every"]) if case["every"] else 0)
    return {"bytes": one(n, depth, meas, case["shots"]), "flops": 0}


def exact(case, seed):
    """Every output is a bit: there is no rounding, and nothing to compare in 64 bits."""
    return None
