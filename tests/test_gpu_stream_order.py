"""Uploads that a propagation makes on its first run: the handles' streams do not wait for the default stream, so the
data must be ordered on the stream that reads it.  A fresh handle's first run equals a repeated one bit for bit."""
import os
import re

import numpy as np
import pytest

import qhfpe_inputs as qi

API = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1706_09590_gb300", "csrc", "qhfpe_api.cu")


def test_no_upload_on_the_default_stream():
    """cudaMemcpy from pageable memory may return before the data has arrived, and orders nothing but the default stream."""
    with open(API) as f:
        plain = re.findall(r"\bcudaMemcpy\([^;]*;", f.read())
    assert not [c for c in plain if "HostToDevice" in c]


def _handles(n, reps=1, persistent=False, nq=120, n_p=64):
    from paper_1706_09590_gb300 import Propagator
    out = []
    for k in range(n):
        m = qi.harmonic_two_state(nq=nq + k, n_p=n_p, depth=1)
        P = Propagator(m, qi.u_table(m), precision="mixed", n_replicas=reps)
        P.set_persistent(persistent)
        out.append(P)
    return out


def _fill(P):
    for r in range(P.n_replicas):
        P.set_state(qi.random_state(P.model, seed=5 + r, hermitian=True), r)


@pytest.mark.gpu
@pytest.mark.parametrize("persistent", [False, True])
def test_first_run_equals_the_second(persistent):
    for P in _handles(4, persistent=persistent):
        out = []
        for _ in range(2):
            _fill(P)
            P.step(2)
            out.append(P.get_state(0))
        P.close()
        assert np.array_equal(out[0], out[1])


@pytest.mark.gpu
def test_first_batch_run_and_a_member_alone():
    """A batch runs on its first member's stream; a member stepped alone afterwards finds its tables complete."""
    from paper_1706_09590_gb300 import Batch
    hs = _handles(3, nq=40, n_p=32)
    for P in hs:
        _fill(P)
    b = Batch(hs)
    b.step(2)
    first = [P.get_state(0) for P in hs]
    for P in hs:
        _fill(P)
    hs[2].step(2)
    alone = hs[2].get_state(0)
    _fill(hs[2])
    b.step(2)
    again = [P.get_state(0) for P in hs]
    b.close()
    for P in hs:
        P.close()
    assert np.array_equal(alone, first[2])
    for x, y in zip(first, again):
        assert np.array_equal(x, y)
