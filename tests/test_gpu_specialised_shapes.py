"""Specialised kernels on the library's own tile where most qubits of a part
are controls and phases outside it, against the oracle."""
import pytest

from oracle import sim
from tests.gpu_util import TOL, max_abs, random_state, run_gpu
from tests.test_specialise_shapes import few_in_the_tile

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["qft", "cp", "ctl"])
@pytest.mark.parametrize("n", [12, 15, 17, 20])
def test_largest_part_in_the_tile(kind, n):
    g = few_in_the_tile(kind, n)
    psi = random_state(n, n)
    ref = sim.run(n, g, psi)
    for precision, method, k in (("c64", "dfs", 12), ("c64", "dagp", 11), ("c64", "nat", min(n, 13)),
                                 ("c128", "dagp", 12), ("c128df", "dfs", 12)):
        out = run_gpu(n, g, method=method, k=k, precision=precision, psi=psi, jit=True)
        assert max_abs(out, ref) <= TOL[precision], (precision, method, k)
