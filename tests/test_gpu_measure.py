"""Probabilities, norms and summaries on the GPU against FP64 arithmetic on
the host, at the edges of the FP32 kernels' range: one chunk and less, pairs
that are not aligned for vector stores, amplitudes too small or too large for
the split, equal maxima."""
import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import native, random_state

pytestmark = pytest.mark.gpu


def _state(api, psi, precision):
    n = int(np.log2(len(psi)))
    st = api.State(n, precision)
    dt = torch.complex64 if precision == "c64" else torch.complex128
    st.upload(torch.from_numpy(np.ascontiguousarray(psi)).to(dt).pin_memory())
    a = st.copy_to_host().numpy().astype(np.complex128)
    return st, a.real * a.real + a.imag * a.imag


def _check(st, p):
    # a float rounding of the FP64 value; a float too large is infinite, one
    # below the normal range is off by a unit of the denormals
    tol = np.abs(p) * 2.0 ** -23.9 + 2.0 ** -148
    for shift in (0, 1):   # 1: an output that is only aligned to 4 bytes
        out = torch.empty(len(p) + shift, dtype=torch.float32, device="cuda")[shift:]
        norm = st.probs(out)
        got = out.cpu().numpy().astype(np.float64)
        with np.errstate(over="ignore"):
            big = np.isinf(p.astype(np.float32))
        assert np.array_equal(np.isinf(got), big)
        assert (np.abs(got - p)[~big] <= tol[~big]).all()
        assert abs(norm - p.sum()) <= 1e-13 * p.sum()
    out = torch.empty(len(p), dtype=torch.float64, device="cuda")
    st.probs(out, fp64=True)
    assert (np.abs(out.cpu().numpy() - p) <= 1e-14 * p + 1e-300).all()
    norm, p0, am, pm = st.summary()
    assert am == int(np.argmax(p))
    assert abs(norm - p.sum()) <= 1e-13 * p.sum()
    assert abs(p0 - p[0]) <= 1e-14 * p[0] and abs(pm - p.max()) <= 1e-14 * p.max()


@pytest.mark.parametrize("precision", ["c64", "c128", "c128df"])
@pytest.mark.parametrize("n", [1, 9, 10, 11, 12, 17, 21])
def test_random_states(precision, n):
    _, api = native()
    st, p = _state(api, random_state(n, 5 + n), precision)
    _check(st, p)
    _check(st, p)   # the reduction's ticket is back at zero
    st.close()


@pytest.mark.parametrize("precision", ["c64", "c128df"])
def test_outside_the_split(precision):
    """Amplitudes around the split's limits, zeros, and a largest probability
    that overflows a float."""
    _, api = native()
    psi = random_state(13, 1)
    r = synth.SplitMix64(2)
    for s in (1e-25, 2.0 ** -50, 2.0 ** -51, 0.0, 2.0 ** 59, 2.0 ** 60, 2.0 ** 63):
        for _ in range(40):
            psi[r.randint(1 << 13)] *= s
    st, p = _state(api, psi, precision)
    _check(st, p)
    st.close()


@pytest.mark.parametrize("precision", ["c64", "c128", "c128df"])
def test_equal_probabilities(precision):
    """Every probability the same, then two equal maxima: the smallest index."""
    _, api = native()
    psi = np.full(1 << 14, 2.0 ** -7, dtype=np.complex128)
    st, p = _state(api, psi, precision)
    _check(st, p)
    assert st.summary()[2] == 0
    st.close()
    psi[[9001, 777, 16000]] *= 1.5
    st, p = _state(api, psi, precision)
    _check(st, p)
    assert st.summary()[2] == 777
    st.close()


def test_batch_probs_alignment_and_norms():
    native()
    from paper_2205_06973_gb300.batch import Batch
    circs = [synth.batch_circuit(i) for i in (4, 5)] + [(10, synth.qft(10)), (14, synth.layered(14, 3, 1))]
    b = Batch(circs, method="dagp", k=8)
    b.run(sync=True)
    p = np.concatenate([np.abs(b.state_host(i).numpy().astype(np.complex128)) ** 2 for i in range(len(circs))])
    for shift in (0, 1):
        out = torch.empty(b.total + shift, dtype=torch.float32, device="cuda")[shift:]
        torch.cuda.synchronize()
        _, norms = b.probs(out)
        assert (np.abs(out.cpu().numpy() - p) <= p * 2.0 ** -23.9 + 2.0 ** -148).all()
        for i in range(len(circs)):
            assert abs(norms[i] - p[b.offsets[i]:b.offsets[i + 1]].sum()) <= 1e-13
    only = b.probs(torch.zeros(b.total, dtype=torch.float32, device="cuda"), norms=False)
    b.sync()
    assert only[1] is None
    b.close()


def test_more_states_than_result_slots():
    """The 65th live state that measures copies its results."""
    _, api = native()
    n = 6
    states = []
    for i in range(66):
        st = api.State(n)
        st.set_basis(i % 64)
        states.append(st)
    for i, st in enumerate(states):
        assert st.summary() == (1.0, float(i % 64 == 0), i % 64, 1.0)
        p = torch.empty(1 << n, device="cuda")
        assert st.probs(p) == 1.0 and int(p.argmax()) == i % 64
    states[3].close()
    assert states[65].summary() == (1.0, 0.0, 1, 1.0)
    for st in states:
        st.close()
