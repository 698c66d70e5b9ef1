"""Circuits on fewer than 10 qubits: the one-launch kernel against the oracle
for every gate kind and size, and a first apply inside a stream capture."""
import numpy as np
import pytest
import torch

from oracle import sim
from tests.gpu_util import TOL, max_abs, native, random_state, run_gpu
from tests.test_gpu_parity import _all_kinds

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["c64", "c128"])
@pytest.mark.parametrize("n", range(1, 10))
def test_all_gate_kinds(precision, n):
    """63 to 130 gates: less than, exactly, and more than one staged block."""
    for G in (1, 64, 130):
        if n == 1:
            g = [(name, (0,), th) for name, q, th in _all_kinds(2, 3 * G, n + G) if len(q) == 1][:G]
        else:
            g = _all_kinds(n, G, n + G)
        psi = random_state(n, 7 + n)
        out = run_gpu(n, g, method="dagp", k=2 if n > 1 else 1, precision=precision, psi=psi)
        assert max_abs(out, sim.run(n, g, psi)) <= TOL[precision], G


def test_first_apply_inside_a_capture():
    _, api = native()
    n = 7
    g = _all_kinds(n, 40, 3)
    plan = api.Plan(g, n, "dagp", 4)
    psi = random_state(n, 1)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        st = api.State(n, "c128", stream=stream)
        st.upload(torch.from_numpy(psi).pin_memory())
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            st.apply(plan)
        graph.replay()
        graph.replay()
        out = st.copy_to_host().numpy()
    ref = sim.run(n, g, sim.run(n, g, psi))
    assert max_abs(out, ref) <= TOL["c128"]
    st.apply(plan, sync=True)   # outside: uploads and takes the one-launch kernel
    assert max_abs(st.copy_to_host().numpy(), sim.run(n, g, ref)) <= TOL["c128"]
    st.close()
    plan.close()
