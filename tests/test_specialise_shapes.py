"""The tile and register bits that the library chooses for specialised kernels
hold the plan's largest part, also where most of its qubits are controls and
need no place in the tile (host only: the kernels compile with NVRTC)."""
import pytest

import synth


def few_in_the_tile(kind, n):
    """Parts of many qubits of which few are acted on other than as phases and
    controls; "qft": one phase and control at a time."""
    r = synth.SplitMix64(n)
    if kind == "qft":
        return synth.qft(n)
    if kind == "cp":
        return [("CP", (a, (a + 1 + r.randint(n - 1)) % n), r.angle()) for a in range(n) for _ in range(4)]
    g = []   # H and CX on one qubit under all the others
    for i in range(4 * n):
        g += [("H", (0,), 0.0), (("CX", "CZ", "CP")[i % 3], (1 + i % (n - 1), 0), r.angle())]
    return g


@pytest.mark.parametrize("kind,method,n,k", [("qft", "dfs", 15, 12), ("qft", "dfs", 17, 12), ("cp", "dagp", 14, 12),
                                             ("ctl", "dagp", 14, 12), ("ctl", "nat", 12, 12), ("cp", "beam", 17, 13),
                                             ("qft", "nat", 13, 13), ("ctl", "dfs", 16, 11), ("cp", "dagp", 20, 12)])
def test_default_shape_holds_the_largest_part(kind, method, n, k):
    from paper_2205_06973_gb300 import build
    build.build()
    from paper_2205_06973_gb300 import api
    plan = api.Plan(few_in_the_tile(kind, n), n, method, k)
    for precision in ("c64", "c128", "c128df") if k <= 12 else ("c64",):
        assert plan.specialise(precision, load=False) > 0.0
    plan.close()
