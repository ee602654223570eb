"""Every instantiation of the FP64 stage (np 32 to 256, one to three states) against the oracle: right-hand sides, and steps
as single launches, in a batch of two different members, and in the persistent kernel; linear and nonlinear coupling."""
import numpy as np
import pytest

import oracle
import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


def _model(S, n_p, nq, c2=0.0):
    pr = (-8.0, 8.0) if n_p < 128 else (-16.0, 16.0)
    if S == 1:
        m = qi.single_state(lambda q: 0.5 * q * q, nq=nq, n_p=n_p, pr=pr, depth=2, closure=0)
    elif S == 2:
        m = qi.photoisomerization_two_state(nq=nq, n_p=n_p, pr=pr, depth=1, n_matsubara=1)
    else:
        m = qi.three_state(nq=nq, n_p=n_p, depth=1, n_matsubara=1)
    m["dt"] = 1e-4
    if c2:
        m["v_c2"] = c2
    return m


def _P(m):
    from paper_1706_09590_gb300 import Propagator
    P = Propagator(m, qi.u_table(m), precision="fp64")
    P.set_state(qi.random_state(m, seed=17, hermitian=True))
    return P


@pytest.mark.parametrize("S", [1, 2, 3])
@pytest.mark.parametrize("n_p", [32, 64, 128, 256])
@pytest.mark.parametrize("c2", [0.0, 0.05])
def test_rhs_and_steps(S, n_p, c2, monkeypatch):
    for tile in ("1", "3", "4"):
        monkeypatch.setenv("QHFPE_TILE_ROWS", tile)
        m = _model(S, n_p, 9, c2)
        P, O = _P(m), oracle.Oracle(m)
        W = P.get_state(0)
        assert rel(P.apply_rhs(0), O.rhs(W)) < 1e-12  # (as elsewhere)
        P.step(2)
        assert rel(P.get_state(0), O.step(W, 2)[0]) < 1e-12
        P.close()


@pytest.mark.parametrize("S", [1, 2, 3])
@pytest.mark.parametrize("n_p", [32, 64, 128, 256])
@pytest.mark.parametrize("c2", [0.0, 0.05])
def test_batch_and_persistent(S, n_p, c2):
    from paper_1706_09590_gb300 import Batch
    ms = [_model(S, n_p, 10, c2), _model(S, n_p, 7, c2)]
    ref = []
    for persistent in (False, True):
        Ps = [_P(m) for m in ms]
        W = [P.get_state(0) for P in Ps]
        if persistent:
            for P in Ps:
                P.set_persistent(True)
                P.step(2)
        else:
            B = Batch(Ps)
            B.step(2)
            ref = [oracle.Oracle(m).step(w, 2)[0] for m, w in zip(ms, W)]
            B.close()
        for P, r in zip(Ps, ref):
            assert rel(P.get_state(0), r) < 1e-12
            P.close()
