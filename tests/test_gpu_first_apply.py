"""Statistics and apply share one compiled program: a server asks for the
statistics of a large request's plan on a planner thread, and its scheduler
thread must not compile the plan again at the apply."""
import time

import pytest

import synth
from tests.gpu_util import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method,k,tc", [("beam", 6, True), ("beam", 6, 2), ("beam", 7, True), ("beam", 10, False)])
def test_apply_after_stats_does_not_compile_again(method, k, tc):
    """The compilation takes tens of milliseconds; the first apply after it
    uploads a few megabytes."""
    _, api = native()
    n = 22
    st = api.State(n)
    compile_s, apply_s = [], []
    for i in range(4):   # the first loads the kernels
        plan = api.Plan(synth.layered(n, 40, 7 + i, two_q=("CX", "CZ")), n, method, k, dfs_trials=8)
        st.set_basis(0)
        st.sync()
        t0 = time.perf_counter()
        stats = plan.stats("c64", tc=tc)
        t1 = time.perf_counter()
        st.apply(plan, tc=tc)
        t2 = time.perf_counter()
        st.sync()
        assert stats["passes"] > 0
        if i:
            compile_s.append(t1 - t0)
            apply_s.append(t2 - t1)
        plan.close()
    st.close()
    assert min(apply_s) < 0.5 * min(compile_s), (apply_s, compile_s)
