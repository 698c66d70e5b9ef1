"""Circuits on fewer than 10 qubits need nothing of the plan after the call: a
plan dropped behind an asynchronous apply, a captured graph replayed after its
plan is closed; and lists longer than one launch takes."""
import numpy as np
import pytest
import torch

from oracle import sim
from tests.gpu_util import TOL, max_abs, native, random_state, run_gpu
from tests.test_gpu_parity import _all_kinds

pytestmark = pytest.mark.gpu


def _state(api, psi, precision, stream):
    st = api.State(int(np.log2(len(psi))), precision, stream=stream)
    st.upload(torch.from_numpy(psi).to(torch.complex64 if precision == "c64" else torch.complex128).pin_memory())
    st.sync()
    return st


@pytest.mark.parametrize("precision", ["c64", "c128"])
def test_plan_dropped_behind_its_apply(precision):
    _, api = native()
    n = 8
    stream = torch.cuda.Stream()
    psi = random_state(n, 1)
    st = _state(api, psi, precision, stream)
    big = api.State(24, stream=stream)   # work in front, so that the applies are still queued
    long = api.Plan(_all_kinds(24, 200, 1), 24, "dagp", 8)
    big.set_basis(0)
    ref = psi
    big.apply(long)
    for i in range(20):
        g = _all_kinds(n, 60, i)
        st.apply(api.Plan(g, n, "dagp", 4))
        ref = sim.run(n, g, ref)
    out = st.copy_to_host().numpy()
    assert max_abs(out, ref) <= 10 * TOL[precision]
    st.close()
    big.close()


def test_graph_outlives_its_plan():
    _, api = native()
    n = 7
    g = _all_kinds(n, 50, 2)
    psi = random_state(n, 2)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        st = _state(api, psi, "c128", stream)
        plan = api.Plan(g, n, "dagp", 4)
        st.apply(plan)   # not the first apply of the plan
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            st.apply(plan)
        plan.close()
        other = api.Plan(_all_kinds(n, 50, 3), n, "dagp", 4)
        rest = _state(api, psi, "c128", stream)
        rest.apply(other, sync=True)
        graph.replay()
        out = st.copy_to_host().numpy()
    assert max_abs(out, sim.run(n, g, sim.run(n, g, psi))) <= TOL["c128"]


@pytest.mark.parametrize("precision,ops", [("c64", 80), ("c64", 81), ("c64", 256), ("c64", 257), ("c64", 640),
                                           ("c64", 641), ("c64", 1300), ("c128", 48), ("c128", 49), ("c128", 152),
                                           ("c128", 153), ("c128", 384), ("c128", 385), ("c128", 800)])
def test_list_lengths(precision, ops):
    """ops records: alternating phases and one-qubit gates that do not fuse."""
    n = 6
    g = []
    while len(g) < ops:
        i = len(g)
        g.append(("CP", (i % n, (i + 1) % n), 0.1 + i) if i % 2 else ("RX", ((i // 2) % n, ), 0.2 + i))
        if len(g) < ops and i % 2:
            g.append(("CZ", (i % n, (i + 2) % n), 0.0))
    psi = random_state(n, ops)
    out = run_gpu(n, g, method="dagp", k=4, precision=precision, psi=psi)
    assert max_abs(out, sim.run(n, g, psi)) <= TOL[precision]
