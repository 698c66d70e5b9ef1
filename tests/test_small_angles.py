"""Many parts of small rotations in complex128 (Trotter steps): a part's factor
is within 1e-13 of 1, but not a phase; dropping it would grow the norm by that
much a part. The generated kernels, built for the host."""
import numpy as np
import pytest

from oracle import sim
from tests.test_specialise_host import _psi, pytestmark, run_host  # noqa: F401


def trotter(parts, angle):
    """Parts of four qubits (nat order, k = 4): rotations by a small angle on
    all, then phases that merge into one diagonal."""
    g = []
    for p in range(parts):
        q = [4 * (p % 2) + i for i in range(4)]
        g += [("RX" if (i + p) % 2 else "RY", (x,), angle * (1 + i % 3)) for i, x in enumerate(q)]
        g += [("CP", (q[i], q[i + 1]), 0.2 + i) for i in range(3)]
        g += [("RZ", (x,), 0.3 + 0.1 * i) for i, x in enumerate(q)]
    return g


@pytest.mark.parametrize("angle", [2e-7, 3.5e-7])
def test_norm_of_small_rotations_host(angle):
    n, parts = 10, 60
    g = trotter(parts, angle)
    psi = _psi(n, 6)
    out = run_host(n, g, "nat", 4, "c128", psi=psi)
    # each gate rounds an amplitude's parts to 2^-53 a few times
    tol = len(g) * 2.0 ** -52
    assert abs(np.vdot(out, out).real / np.vdot(psi, psi).real - 1.0) <= tol
    assert np.abs(out - sim.run(n, g, psi)).max() <= tol
