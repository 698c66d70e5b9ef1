"""Long circuits on few targets: hundreds of gates whose factors (1/sqrt2 of an
H, the largest entry of a rotation) the planner gathers stay in one register
phase, so the factors must be applied within it before they or the
unnormalised amplitudes leave the range of a float. The generated kernels,
built for the host, against the oracle."""
import numpy as np
import pytest

import synth
from oracle import sim
from tests.test_specialise_host import TOL, _psi, pytestmark, run_host  # noqa: F401


def few_targets(n, steps, seed):
    """Steps of H, RX, RY and a general one-qubit run on three qubits with CX
    between them and phases from changing other qubits."""
    r = synth.SplitMix64(seed)
    g = []
    for i in range(steps):
        g += [("H", (q,), 0.0) for q in range(3)]
        g += [("CX", (0, 1), 0.0), ("CX", (1, 2), 0.0), ("T", (2,), 0.0),
              ("CP", (3 + i % (n - 3), i % 3), r.angle())]
        if i % 4 == 1:
            g += [(name, (i % 3,), r.angle()) for name in ("RX", "RZ", "RY", "H")]
        if i % 4 == 3:
            g += [("RX", (0,), 1.5), ("CZ", (0, 1), 0.0), ("RY", (1,), 1.6)]
    return g


def ancilla(n, reps):
    return [x for i in range(reps) for x in (("H", (0,), 0.0), ("CP", (1 + i % (n - 1), 0), 0.3 + i))]


@pytest.mark.parametrize("precision", ["c64", "c128", "c128df"])
@pytest.mark.parametrize("steps", [30, 120])
def test_few_targets_host(precision, steps):
    n = 10
    g = few_targets(n, steps, steps)
    psi = _psi(n, 3)
    out = run_host(n, g, "dagp", n, precision, psi=psi)
    assert np.abs(out - sim.run(n, g, psi)).max() <= TOL[precision]


def test_one_target_host():
    n = 10
    g = ancilla(n, 400)
    psi = _psi(n, 4)
    out = run_host(n, g, "dagp", n, "c64", psi=psi)
    assert np.abs(out - sim.run(n, g, psi)).max() <= TOL["c64"]
