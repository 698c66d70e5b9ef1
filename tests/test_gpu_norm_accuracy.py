"""Norms and probabilities on the FP32 pipes have FP64's accuracy: against
exact sums, over states of one to a few amplitudes (where no rounding averages
out) and random ones, complex64 and double-float."""
import math

import numpy as np
import pytest
import torch

from tests.gpu_util import native, random_state

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _floats(psi, precision):
    """The amplitudes' components as the device holds them: rows of floats
    whose sum is the component."""
    v = np.ascontiguousarray(psi).view(np.float64)
    hi = v.astype(np.float32)
    if precision == "c64":
        return hi.astype(np.float64)[None]
    return np.stack((hi, (v - hi).astype(np.float32))).astype(np.float64)


def _exact(f):
    """Sum of the squared components: products of floats are exact in FP64,
    their sum is fsum's."""
    terms = [f[0] * f[0]] + ([2.0 * f[0] * f[1], f[1] * f[1]] if len(f) > 1 else [])
    return math.fsum(x for t in terms for x in t[t != 0.0])


def _errors(st, psi, precision):
    dt = torch.complex64 if precision == "c64" else torch.complex128
    st.upload(torch.from_numpy(psi).to(dt).pin_memory())
    ref = _exact(_floats(psi, precision))
    out = torch.empty(len(psi), dtype=torch.float32, device="cuda")
    return [abs(x - ref) / ref for x in (st.probs(out), st.probs(), st.summary()[0])]


def sparse(n, m, r):
    psi = np.zeros(1 << n, dtype=np.complex128)
    at = r.integers(0, 1 << n, m)
    psi[at] = r.normal(size=m) + 1j * r.normal(size=m)
    return psi * 2.0 ** float(r.integers(-12, 4))


@pytest.mark.parametrize("precision", ["c64", "c128df"])
@pytest.mark.parametrize("n,m", [(11, 1), (12, 3), (14, 10)])
def test_few_amplitudes(precision, n, m):
    """A thread's sum is joined with three roundings, and each further
    nonzero thread adds one or two."""
    _, api = native()
    st = api.State(n, precision)
    r = np.random.default_rng(n)
    for _ in range(64):
        assert max(_errors(st, sparse(n, m, r), precision)) <= (3 + 2 * m) * U
    st.close()


@pytest.mark.parametrize("precision", ["c64", "c128df"])
@pytest.mark.parametrize("n", [11, 13, 17, 20])
def test_random_states(precision, n):
    """At most 8 additions of a thread's sums, 5 of a warp, 8 of a block, 3 + 8
    of the blocks."""
    _, api = native()
    st = api.State(n, precision)
    for seed in range(4):
        assert max(_errors(st, random_state(n, seed), precision)) <= 32 * U
    st.close()


def test_batch_norms():
    native()
    from paper_2205_06973_gb300.batch import Batch
    r = np.random.default_rng(5)
    for _ in range(8):
        b = Batch([(n, [("RY", (q,), float(r.uniform(0, 6))) for q in range(2)]) for n in (10, 11, 13)],
                  method="dagp", k=8)
        b.run(sync=True)
        _, norms = b.probs()
        for i in range(3):
            a = b.state_host(i).numpy().view(np.float32).astype(np.float64)
            ref = math.fsum(x * x for x in a[a != 0.0])
            assert abs(norms[i] - ref) / ref <= 11 * U   # four amplitudes
        b.close()
