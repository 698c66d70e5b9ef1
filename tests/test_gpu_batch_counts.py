"""What a batch reports of itself (sv_batch_info), circuits without gates among
those that run on one CTA."""
import numpy as np
import pytest

import synth
from oracle import sim
from tests.gpu_util import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(10,), (12, 10, 11)])
def test_only_empty_circuits(sizes):
    native()
    from paper_2205_06973_gb300.batch import Batch
    b = Batch([(n, []) for n in sizes], method="dagp", k=8)
    b.run(sync=True)
    info = b.info()
    assert info["items"] == 0 and info["parts"] == 0
    probs, norms = b.probs()
    p = probs.cpu().numpy()
    assert p.sum() == len(sizes) and all(p[o] == 1.0 for o in b.offsets[:-1]) and (np.asarray(norms) == 1.0).all()
    b.close()


def test_counts_of_a_mixed_batch():
    native()
    from paper_2205_06973_gb300.batch import Batch
    circs = [(10, []), (11, synth.layered(11, 4, 1)), (14, synth.layered(14, 4, 2)), (12, []), (12, synth.qft(12))]
    b = Batch(circs, method="dagp", k=8, tiles_per_item=4)
    b.run(sync=True)
    parts = [p.export()[1] for p in b.plans]
    info = b.info()
    assert info["parts"] == sum(parts) - parts[0] - parts[3] and parts[0] == parts[3] == 0
    assert info["items"] == 2 + parts[2] * (32 // 4)   # one CTA each, 2^5 tiles in fours
    for i, (n, g) in enumerate(circs):
        assert np.abs(b.state_host(i).numpy() - sim.run(n, g)).max() <= 1e-5, i
    b.close()
