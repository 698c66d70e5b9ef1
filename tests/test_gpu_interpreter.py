"""The op decoder and the default shapes against the oracle where they change:
whole circuits on one tile (10 to 13 qubits) with programs of several windows
and more unnormalised gates than a part's factor may gather, complex128 tiles
down to 2^8, specialised kernels on the library's tile and register bits, and
a batch's circuits of at most 12 qubits (one CTA each) beside larger ones."""
import numpy as np
import pytest
import torch

import synth
from oracle import sim
from tests.gpu_util import TOL, max_abs, native, random_state, run_gpu
from tests.test_gpu_parity import _all_kinds

pytestmark = pytest.mark.gpu


def _long(n, seed):
    """Every gate kind, then enough layers that the program fills several
    windows (8 KiB) and holds over a hundred H and rotations."""
    return _all_kinds(n, 250, seed) + synth.layered(n, 24, seed, two_q=("CX", "CZ")) + synth.param(n, 3, seed) \
        + _all_kinds(n, 60, seed + 1)


@pytest.mark.parametrize("precision", ["c64", "c128"])
@pytest.mark.parametrize("n", [10, 11, 12, 13, 14])
def test_default_tile(n, precision):
    """k from 2 to the qubit count: tiles of 2^8 and up for complex128."""
    g = _long(n, n)
    psi = random_state(n, n)
    ref = sim.run(n, g, psi)
    for method, k in (("nat", 2), ("dagp", 8), ("dfs", 9), ("beam", min(n, 12))):
        out = run_gpu(n, g, method=method, k=k, precision=precision, psi=psi)
        assert max_abs(out, ref) <= TOL[precision], (method, k)


@pytest.mark.parametrize("precision", ["c64", "c128"])
def test_program_of_several_windows_over_several_tiles(precision):
    n = 15
    g = _long(n, 5) * 2
    psi = random_state(n, 6)
    ref = sim.run(n, g, psi)
    out = run_gpu(n, [x for x in g if max(x[1]) < 11], method="nat", k=11, precision=precision, psi=psi, tile=11)
    assert max_abs(out, sim.run(n, [x for x in g if max(x[1]) < 11], psi)) <= TOL[precision]
    out = run_gpu(n, g, method="dagp", k=10, precision=precision, psi=psi)
    assert max_abs(out, ref) <= TOL[precision]


@pytest.mark.parametrize("precision", ["c64", "c128", "c128df"])
@pytest.mark.parametrize("n", [10, 12, 16, 18, 20])
def test_specialised_default_shape(n, precision):
    g = _all_kinds(n, 120, n) + synth.layered(n, 3, n, two_q=("CX", "CZ"))
    psi = random_state(n, 2 * n)
    ref = sim.run(n, g, psi)
    for method, k in (("dagp", 7), ("beam", 10)):
        out = run_gpu(n, g, method=method, k=k, precision=precision, psi=psi, jit=True)
        assert max_abs(out, ref) <= TOL[precision], (method, k)


@pytest.mark.parametrize("dense", [0, 13])
def test_batch_of_small_and_large(dense):
    native()
    from paper_2205_06973_gb300.batch import Batch
    circs = [(n, _long(n, n)) for n in (12, 10, 11)] + [(14, synth.layered(14, 6, 1)), (10, synth.qft(10)),
                                                        (13, synth.param(13, 5, 2)), (12, [])]
    b = Batch(circs, method="dagp", k=8, dense_min_qubits=dense)
    b.run(sync=True)
    for i, (n, g) in enumerate(circs):
        out = b.state_host(i).numpy().astype(np.complex128)
        assert np.abs(out - sim.run(n, g)).max() <= 1e-5, i
    b.reset()
    b.run(sync=True)
    b.run(sync=True)
    n, g = circs[2]
    out = b.state_host(2).numpy().astype(np.complex128)
    assert np.abs(out - sim.run(n, g, sim.run(n, g))).max() <= 1e-5
    info = b.info()
    assert info["items"] > 0 and info["parts"] >= len(circs) - info["dense_circuits"] - 1
    b.close()
    torch.cuda.synchronize()


def _cx_net(n, depth, seed):
    """Runs of CX (chains both ways, fans, random pairs, onto and off the
    lowest five qubits), SWAPs among them, separated by gates that do and do
    not commute with a CX on either qubit."""
    rng = np.random.default_rng(seed)
    g = [("H", (q,), 0.0) for q in range(n)]
    for _ in range(depth):
        kind = int(rng.integers(4))
        if kind == 0:
            g += [("CX", (q, q + 1), 0.0) for q in range(n - 1)]
        elif kind == 1:
            g += [("CX", (q + 1, q), 0.0) for q in reversed(range(n - 1))]
        elif kind == 2:
            c = int(rng.integers(n))
            g += [("CX", (c, q), 0.0) for q in range(n) if q != c]
        for _ in range(n):
            a, b = (int(x) for x in rng.choice(n, 2, replace=False))
            g.append(("SWAP" if rng.random() < 0.1 else "CX", (a, b), 0.0))
        for q in rng.choice(n, n // 3, replace=False):
            name = ("RZ", "RX", "T", "X", "H", "RY")[int(rng.integers(6))]
            g.append((name, (int(q),), float(rng.uniform(0, 6))))
    return g


@pytest.mark.parametrize("precision", ["c64", "c128", "c128df"])
@pytest.mark.parametrize("n", [10, 13, 16])
def test_cx_at_the_ends_of_phases(n, precision):
    g = _cx_net(n, 8, n)
    psi = random_state(n, 3 * n)
    ref = sim.run(n, g, psi)
    for method, k, tile in (("nat", 8, 10), ("dagp", 7, 0), ("beam", 9, 0), ("dfs", 6, 11)):
        out = run_gpu(n, g, method=method, k=k, precision=precision, psi=psi, tile=min(tile, n))
        assert max_abs(out, ref) <= TOL[precision], (method, k, tile)
