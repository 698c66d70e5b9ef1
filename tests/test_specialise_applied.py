"""What the statistics, flop counts and sources of a plan describe with
SV_FLAG_SPECIALISE: the program that an apply runs, on the library's tile and
register bits, with parts cut and joined and qubits outside the tile. Its
kernels, built for the host, against the oracle."""
import re

import numpy as np
import pytest

import synth
from oracle import sim
from tests import test_specialise_host as host
from tests.test_gpu_parity import _all_kinds
from tests.test_specialise_host import pytestmark  # noqa: F401


@pytest.fixture
def applied(monkeypatch):
    """api with plans that describe the specialised apply."""
    api = host._api()

    class Applied(api.Plan):
        def stats(self, *a, **k):
            return super().stats(*a, **k, jit=True)

        def source(self, *a, **k):
            return super().source(*a, **k, jit=True)

        def flops(self, *a, **k):
            return super().flops(*a, **k, jit=True)

    monkeypatch.setattr(api, "Plan", Applied)
    return api


CASES = [("qft", 13, "beam", 12), ("qft", 15, "dfs", 12), ("layered", 13, "beam", 9), ("kinds", 12, "dagp", 8),
         ("param", 12, "dfs", 7)]


def _gates(kind, n):
    return {"qft": lambda: synth.qft(n), "layered": lambda: synth.layered(n, 8, 3, two_q=("CX", "CZ")),
            "kinds": lambda: _all_kinds(n, 200, 5), "param": lambda: synth.param(n, 4, 2)}[kind]()


@pytest.mark.parametrize("precision", ["c64", "c128", "c128df"])
@pytest.mark.parametrize("kind,n,method,k", CASES)
def test_applied_kernels_host(applied, kind, n, method, k, precision):
    g = _gates(kind, n)
    psi = host._psi(n, 7)
    out = host.run_host(n, g, method, k, precision, psi=psi)
    assert np.abs(out - sim.run(n, g, psi)).max() <= host.TOL[precision]


@pytest.mark.parametrize("kind,n,method,k", CASES + [("qft", 24, "beam", 12), ("layered", 22, "beam", 9)])
def test_statistics_are_of_the_sources(applied, kind, n, method, k):
    for precision in ("c64", "c128", "c128df"):
        plan = applied.Plan(_gates(kind, n), n, method, k)
        st = plan.stats(precision)
        src = [plan.source(i, precision) for i in range(st["passes"])]
        with pytest.raises(Exception):
            plan.source(st["passes"], precision)
        # one gather from shared memory per phase
        assert sum(len(re.findall(r"a\[i\] = cur\[", s)) for s in src) == st["phases"]
        products = sum(len(re.findall(r"op_p<NR|op_prot<NR", s)) for s in src)   # a complex product on half each
        assert plan.flops(precision)[0] >= 3.0 * products * 2.0 ** n
        plan.close()


def test_joined_parts_are_fewer(applied):
    """The 24-qubit QFT's parts of phases alone join their neighbours."""
    plan = applied.Plan(synth.qft(24), 24, "beam", 12)
    own = host._api().Plan.__mro__[1].stats(plan, "c64")["passes"]
    assert plan.stats("c64")["passes"] < own == plan.export()[1]
    plan.close()
