"""Long circuits on few targets against the oracle on every gate-list path: a
whole circuit on one CTA (10 to 13 qubits, alone and in a batch), parts of
larger states, and the specialised kernels. Their gates' factors are below the
range of a float several times over."""
import numpy as np
import pytest

from oracle import sim
from tests.gpu_util import TOL, max_abs, native, random_state, run_gpu
from tests.test_long_phases import ancilla, few_targets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["c64", "c128", "c128df"])
@pytest.mark.parametrize("n", [10, 11, 12, 13, 15])
def test_few_targets(n, precision):
    psi = random_state(n, n)
    for g in (few_targets(n, 100, n), ancilla(n, 300)):
        ref = sim.run(n, g, psi)
        for method, k in (("dagp", 4), ("dagp", 8), ("nat", 10)):
            for jit in (False, True):
                out = run_gpu(n, g, method=method, k=k, precision=precision, psi=psi, jit=jit)
                assert max_abs(out, ref) <= TOL[precision], (method, k, jit)


@pytest.mark.parametrize("k", [4, 8])
def test_few_targets_in_a_batch(k):
    native()
    from paper_2205_06973_gb300.batch import Batch
    circs = [(n, few_targets(n, 100, n)) for n in (10, 11, 12, 13)] + [(n, ancilla(n, 300)) for n in (10, 12, 14)]
    b = Batch(circs, method="dagp", k=k)
    b.run(sync=True)
    for i, (n, g) in enumerate(circs):
        out = b.state_host(i).numpy().astype(np.complex128)
        assert max_abs(out, sim.run(n, g)) <= TOL["c64"], i
    b.close()
