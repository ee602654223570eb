"""Cluster-resident propagation over the range of FP32, subnormal values among it, against the launch-per-stage form (the
zeroth tier is FP64 in both: base and update of every stage)."""
import numpy as np
import pytest

import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


# FP32 stages in another order, 3e-6 over some steps as for values of order one; at 1e-40 the stages' values are
# multiples of 2^-149 = 1.4e-45: 7e-6 of a value, in sums of weights up to 130 / 60, a step of 0.01
@pytest.mark.parametrize("scale,tol", [(1e-40, 1e-4), (1e-30, 3e-6), (1e30, 3e-6)])
@pytest.mark.parametrize("n_p", [32, 64])
def test_scaled_states(scale, tol, n_p, monkeypatch):
    from paper_1706_09590_gb300 import Propagator
    m = qi.harmonic_two_state(nq=20, n_p=n_p, depth=2)
    W = qi.random_state(m, seed=81, hermitian=True)
    out = []
    for resident in ("1", "0"):
        monkeypatch.setenv("QHFPE_RESIDENT", resident)
        P = Propagator(m, qi.u_table(m), precision="mixed")
        P.set_state(W * scale)
        P.step(6)
        out.append(P.get_state(0) / scale)
        P.close()
    assert rel(out[0][0], out[1][0]) < tol and rel(out[0], out[1]) < tol
    assert rel(out[0][0], W[0]) > 0.01  # it moved
