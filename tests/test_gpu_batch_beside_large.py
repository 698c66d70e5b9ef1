"""A batch does not wait for the passes that other streams have queued, as a
server has them: two low-priority and four medium-priority streams with large
states, batches on high-priority streams. In a process of its own, since what
the streams share is decided as they are created."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import time
import torch
import synth
from paper_2205_06973_gb300 import api
from paper_2205_06973_gb300.batch import Batch
lo, hi = torch.cuda.Stream.priority_range()
n = 26
plan = api.Plan(synth.layered(n, 20, 1), n, "beam", 6, dfs_trials=4)
large = [api.State(n, stream=torch.cuda.Stream(priority=p)) for p in [lo] * 2 + [lo - 1] * 4]
streams = [torch.cuda.Stream(priority=hi) for _ in range(2)]
for st in large:   # the program is uploaded, the kernels are loaded
    st.set_basis(0)
    st.apply(plan, sync=True, tc=True)
for i in range(6):
    b = Batch([(m, synth.param(m, 6, 10 * i + m)) for m in (10, 11, 12, 14, 16)], method="dagp", k=8,
              stream=streams[i % 2], dense_min_qubits=13)
    b.prepare()
    torch.cuda.synchronize()
    for st in large:
        for _ in range(4):
            st.apply(plan, tc=True)
    t0 = time.perf_counter()
    b.run(sync=True)
    t1 = time.perf_counter()
    torch.cuda.synchronize()
    print("batch", t1 - t0, "backlog", time.perf_counter() - t0)
    b.close()
"""


def test_batch_beside_large_states():
    """The backlog is some 180 ms of passes of 0.2 ms, the batch 0.3 ms."""
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=240)
    assert r.returncode == 0, r.stderr[-2000:]
    rows = [line.split() for line in r.stdout.splitlines() if line.startswith("batch")]
    assert len(rows) == 6
    for _, batch, _, backlog in rows:
        assert float(batch) < 0.3 * float(backlog), rows
