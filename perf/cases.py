"""The work that users of the simulator have it do, as cases to measure.

A case is a dict of plain values. ``kind`` says which entry points it calls:

* ``apply``: a circuit applied to a state the program already holds
  (``State.apply``): ``mode`` "parts" is the default call (gate-list kernels
  with the run-time op decoder; below 10 qubits gate by gate), "jit" the
  kernels specialised for a plan that is kept, "tc" the tensor-core parts.
* ``batch``: many small parameterised circuits in one graph launch, each
  from |0...0> to its probability vector (``Batch``).
* ``probs``: the probability vector and norm of a state (``State.probs``).
* ``summary``: norm and most likely basis state without a probability vector
  (``State.summary``), what a server returns for a request.

Circuits are the repository's synthetic families (``synth``): random layered
circuits, the QFT, and parameterised ansatz layers. The circuit of an
``apply`` case is fixed by the case (``circuit``); the seed gives the input
state, a normalised random state as it stands in the middle of a computation
(Porter-Thomas distributed probabilities). The seed of a ``batch`` gives the
angles.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import synth
from paper_2205_06973_gb300 import api
from paper_2205_06973_gb300.batch import Batch


def listed():
    return [
        # tutorial and unit-test sized circuit: all of it is launches
        {"name": "gates-8q-c64", "kind": "apply", "family": "param", "n": 8, "depth": 6, "circuit": 11,
         "precision": "c64", "mode": "parts", "method": "dagp", "k": 6},
        # the 14-qubit complex128 layered circuit (840 gates) on the default call
        {"name": "parts-14q-c128", "kind": "apply", "family": "layered", "n": 14, "depth": 40, "circuit": 1,
         "precision": "c128", "mode": "parts", "method": "dagp", "k": 8},
        # a circuit that is run once, so not worth compiling for: the default call, odd size
        {"name": "parts-21q-c64", "kind": "apply", "family": "layered", "n": 21, "depth": 15, "circuit": 12,
         "precision": "c64", "mode": "parts", "method": "beam", "k": 10},
        # variational circuit evaluated again and again, state inside L2
        {"name": "jit-19q-c64", "kind": "apply", "family": "param", "n": 19, "depth": 20, "circuit": 13,
         "precision": "c64", "mode": "jit", "method": "beam", "k": 10},
        # the benchmark's 28-qubit layered circuit (2 GiB state), a third of its depth
        {"name": "jit-28q-c64", "kind": "apply", "family": "layered", "n": 28, "depth": 20, "circuit": 2,
         "precision": "c64", "mode": "jit", "method": "beam", "k": 9},
        # the QFT on a large register (8 GiB state): long diagonal ladders, few passes
        {"name": "jit-30q-qft-c64", "kind": "apply", "family": "qft", "n": 30, "depth": 1, "circuit": 0,
         "precision": "c64", "mode": "jit", "method": "beam", "k": 12},
        # a served medium-sized request: tensor-core parts of at most 6 qubits
        {"name": "tc-23q-c64", "kind": "apply", "family": "param", "n": 23, "depth": 15, "circuit": 14,
         "precision": "c64", "mode": "tc", "method": "beam", "k": 6},
        # full double precision, larger than L2
        {"name": "jit-24q-c128", "kind": "apply", "family": "layered", "n": 24, "depth": 20, "circuit": 15,
         "precision": "c128", "mode": "jit", "method": "dagp", "k": 10},
        # complex128 in double-float arithmetic
        {"name": "jit-25q-c128df", "kind": "apply", "family": "layered", "n": 25, "depth": 10, "circuit": 16,
         "precision": "c128df", "mode": "jit", "method": "beam", "k": 8},
        # uneven parameterised circuits of 10 to 20 qubits, as a batch service collects them
        {"name": "batch-160", "kind": "batch", "count": 160, "n_min": 10, "n_max": 20, "depth_min": 10,
         "depth_max": 50, "circuit": 4},
        # measurement of a 2 GiB state into a probability vector
        {"name": "probs-28q-c64", "kind": "probs", "n": 28, "precision": "c64", "fp64": False},
        # the result of a served request: no probability vector
        {"name": "summary-25q-c64", "kind": "summary", "n": 25, "precision": "c64"},
    ]


def draw(rng):
    """One more case of the same ranges: qubit counts (the logarithm of the
    state) and depths spread over what the tests, the benchmark and the
    serving stream use."""
    kind = rng.choice(("gates", "parts", "parts", "jit", "jit", "jit", "tc", "tc", "qft", "batch", "probs", "summary"))
    circuit = rng.randrange(1 << 20)
    family = rng.choice(("layered", "param"))
    if kind == "gates":
        return {"kind": "apply", "family": family, "n": rng.randint(4, 9), "depth": rng.randint(3, 12),
                "circuit": circuit, "precision": rng.choice(("c64", "c128")), "mode": "parts", "method": "dagp", "k": 4}
    if kind == "parts":
        precision = rng.choice(("c64", "c64", "c128"))
        return {"kind": "apply", "family": family, "n": rng.randint(10, 24 if precision == "c64" else 21),
                "depth": rng.randint(5, 20), "circuit": circuit, "precision": precision, "mode": "parts",
                "method": rng.choice(("dfs", "dagp", "beam")), "k": rng.randint(7, 10)}
    if kind == "jit":
        precision = rng.choice(("c64", "c64", "c128", "c128df"))
        top = {"c64": 28, "c128": 24, "c128df": 25}[precision]
        return {"kind": "apply", "family": family, "n": rng.randint(12, top), "depth": rng.randint(4, 12),
                "circuit": circuit, "precision": precision, "mode": "jit",
                "method": rng.choice(("dfs", "dagp", "beam")), "k": rng.randint(8, 11)}
    if kind == "tc":
        return {"kind": "apply", "family": family, "n": rng.randint(13, 27), "depth": rng.randint(5, 20),
                "circuit": circuit, "precision": "c64", "mode": "tc", "method": rng.choice(("dagp", "beam")),
                "k": rng.randint(5, 6)}
    if kind == "qft":
        return {"kind": "apply", "family": "qft", "n": rng.randint(14, 29), "depth": 1, "circuit": 0,
                "precision": "c64", "mode": "jit", "method": rng.choice(("dagp", "beam")), "k": rng.randint(9, 12)}
    if kind == "batch":
        lo = rng.randint(10, 14)
        return {"kind": "batch", "count": round(16 * 10 ** rng.random()), "n_min": lo, "n_max": rng.randint(lo + 2, 19),
                "depth_min": 10, "depth_max": rng.randint(15, 50), "circuit": circuit}
    precision = rng.choice(("c64", "c64", "c128", "c128df"))
    case = {"kind": kind, "n": rng.randint(10, 28 if precision == "c64" else 27), "precision": precision}
    if kind == "probs":
        case["fp64"] = rng.random() < 0.3
    return case


def _circuit(case):
    n, depth, seed = case["n"], case["depth"], case["circuit"]
    if case["family"] == "qft":
        return synth.qft(n)
    if case["family"] == "param":
        return synth.param(n, depth, seed)
    return synth.layered(n, depth, seed, two_q=("CX", "CZ"))


def _batch_circuits(case, seed):
    """Sizes and depths from the case, angles from the seed."""
    sizes, angles = synth.SplitMix64(case["circuit"]), synth.SplitMix64(seed)
    out = []
    for _ in range(case["count"]):
        n = case["n_min"] + sizes.randint(case["n_max"] - case["n_min"] + 1)
        depth = case["depth_min"] + sizes.randint(case["depth_max"] - case["depth_min"] + 1)
        out.append((n, synth.param(n, depth, 0, rng=angles)))
    return out


def _amplitudes(n, precision, seed):
    """A normalised random state on the GPU, in the layout of a State: complex64
    or complex128, for double-float the float32 quadruples (re.hi, re.lo,
    im.hi, im.lo)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dtype = torch.complex64 if precision == "c64" else torch.complex128
    x = torch.randn(1 << n, dtype=dtype, device="cuda", generator=g)
    x *= 2.0 ** (-n / 2)
    if precision != "c128df":
        return x
    v = torch.view_as_real(x)
    hi = v.float()
    return torch.stack((hi, (v - hi).float()), dim=-1).reshape(1 << n, 4)


@functools.lru_cache(maxsize=None)
def _batch_stream():
    """The stream a service runs its batches on, one after another."""
    return torch.cuda.Stream()


def prepare(case, seed):
    if case["kind"] == "batch":
        batch = Batch(_batch_circuits(case, seed), method="beam", k=9, dense_min_qubits=13, stream=_batch_stream())
        batch.prepare()
        return {"case": case, "batch": batch,
                "out": torch.empty(batch.total, dtype=torch.float32, device="cuda")}
    n, precision = case["n"], case["precision"]
    state = api.State.over(_amplitudes(n, precision, seed), n, precision)
    held = {"case": case, "state": state}
    if case["kind"] == "apply":
        plan = api.Plan(_circuit(case), n, case["method"], min(case["k"], n), dfs_trials=16)
        if case["mode"] == "jit":
            plan.specialise(precision)
        held["plan"] = plan
    elif case["kind"] == "probs":
        held["out"] = torch.empty(1 << n, dtype=torch.float64 if case["fp64"] else torch.float32, device="cuda")
    return held


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.reset()
        batch.run()
        return batch.probs(state["out"], norms=False)[0]
    sv = state["state"]
    if case["kind"] == "probs":
        norm = sv.probs(state["out"], fp64=case["fp64"])
        return [state["out"], norm]
    if case["kind"] == "summary":
        return list(sv.summary())
    sv.apply(state["plan"], tc=case["mode"] == "tc", jit=case["mode"] == "jit")
    return sv.amplitudes()


# floating-point operations of a gate per amplitude of the state: an add per
# component (H), a multiply-add per component (RX, RY, scaled), a complex
# product on half (RZ) or a quarter (CP) of the amplitudes; permutations and
# sign changes none
_FLOPS = {"H": 2.0, "RX": 4.0, "RY": 4.0, "RZ": 3.0, "CP": 1.5, "CX": 0.0, "CZ": 0.0, "SWAP": 0.0}


def work(case):
    if case["kind"] == "batch":
        circuits = _batch_circuits(case, 0)
        amps = sum(1 << n for n, _ in circuits)
        flops = sum(float(1 << n) * sum(_FLOPS[g[0]] for g in gates) for n, gates in circuits)
        return {"bytes": 12.0 * amps, "flops": flops + 3.0 * amps}   # final states and probabilities written
    amps = float(1 << case["n"])
    amp_bytes = 8 if case["precision"] == "c64" else 16
    if case["kind"] == "probs":
        return {"bytes": amps * (amp_bytes + (8 if case["fp64"] else 4)), "flops": 4.0 * amps}
    if case["kind"] == "summary":
        return {"bytes": amps * amp_bytes, "flops": 4.0 * amps}
    return {"bytes": 2.0 * amp_bytes * amps, "flops": amps * sum(_FLOPS[g[0]] for g in _circuit(case))}


# ---------------------------------------------------------------- exact ---
def _matrix(name, theta):
    c, s = math.cos(theta / 2), math.sin(theta / 2)
    return {"H": (math.sqrt(0.5), math.sqrt(0.5), math.sqrt(0.5), -math.sqrt(0.5)),
            "RX": (c, -1j * s, -1j * s, c), "RY": (c, -s, s, c)}[name]


def _apply_exact(psi, gates):
    """The gates applied one after another to the complex128 vector psi, in place."""
    for name, q, theta in gates:
        if len(q) == 1:
            v = psi.view(-1, 2, 1 << q[0])
            a, b = v[:, 0], v[:, 1]
            if name == "RZ":
                a.mul_(complex(math.cos(theta / 2), -math.sin(theta / 2)))
                b.mul_(complex(math.cos(theta / 2), math.sin(theta / 2)))
            else:
                m00, m01, m10, m11 = _matrix(name, theta)
                x = a.clone()
                a.mul_(m00).add_(b, alpha=m01)
                b.mul_(m11).add_(x, alpha=m10)
        else:
            lo, hi = min(q), max(q)
            v = psi.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
            at = (lambda c, t: v[:, t, :, c] if q[1] == hi else v[:, c, :, t])   # control, target bits
            if name == "CX":
                x = at(1, 0).clone()
                at(1, 0).copy_(at(1, 1))
                at(1, 1).copy_(x)
            else:   # CZ
                at(1, 1).neg_()
    return psi


def _param_exact(n, gates):
    """Probabilities of a parameterised ansatz from |0...0>: per layer the
    product RZ RY of every qubit, contracted a few qubits at a time, then the
    CX ladder as one permutation (the new bit q is the XOR of the bits up to q)."""
    y = torch.arange(1 << n, device="cuda")
    source = y ^ ((y << 1) & ((1 << n) - 1))
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1.0
    per_layer = 3 * n - 1
    for at in range(0, len(gates), per_layer):
        layer = gates[at:at + per_layer]
        one = []
        for q in range(n):
            c, s = math.cos(layer[q][2] / 2), math.sin(layer[q][2] / 2)
            z = complex(math.cos(layer[n + q][2] / 2), math.sin(layer[n + q][2] / 2))
            one.append(np.array([[c * z.conjugate(), -s * z.conjugate()], [s * z, c * z]]))
        for q in range(0, n, 5):
            u = np.eye(1)
            for m in one[q:q + 5]:
                u = np.kron(m, u)
            u = torch.from_numpy(u).to(psi.device)
            psi = torch.matmul(u, psi.view(-1, u.shape[0], 1 << q)).reshape(-1)
        psi = psi[source]
    return psi.real.square() + psi.imag.square()


def exact(case, seed):
    if case["kind"] == "batch":
        return torch.cat([_param_exact(n, gates) for n, gates in _batch_circuits(case, seed)])
    x = _amplitudes(case["n"], case["precision"], seed)
    if case["precision"] == "c128df":
        x = torch.view_as_complex(x.double().view(-1, 2, 2).sum(dim=-1))
    x = x.to(torch.complex128)
    if case["kind"] == "apply":
        if case["family"] == "qft":   # sqrt(N) times the inverse DFT
            return torch.fft.ifft(x, norm="ortho")
        return _apply_exact(x, _circuit(case))
    p = x.real.square() + x.imag.square()
    norm = float(p.sum())
    if case["kind"] == "probs":
        return [p, norm]
    return [norm, float(p[0]), None, float(p.max())]
