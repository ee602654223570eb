"""Periodic q axes shorter than the stencils' reach (nq 1, 2, and 3 beside them): rows wrap as often as it takes, in every
stage kernel, against the oracle; and cluster-resident propagations of one q row a block, with periodic q at both np."""
import numpy as np
import pytest

import oracle
import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu


def _P(m, precision, n=1):
    from paper_1706_09590_gb300 import Propagator
    return Propagator(m, qi.u_table(m), precision=precision, n_replicas=n)


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


def _model(kind, nq, n_p):
    pr = (-8.0, 8.0) if n_p < 128 else (-16.0, 16.0)
    if kind == "three":
        m = qi.three_state(nq=nq, n_p=n_p, depth=1, n_matsubara=1)
    elif kind == "one":
        m = qi.single_state(lambda q: 0.5 * q * q, nq=nq, n_p=n_p, pr=pr, depth=2)
    else:
        m = qi.harmonic_two_state(nq=nq, n_p=n_p, pr=(-7.75, 8.25) if kind == "shifted" else pr, depth=2,
                                  closure=0 if kind == "nonlinear" else 1, dt=1e-3)
    m["periodic_q"] = 1
    if kind == "nonlinear":
        m["v_c2"] = 0.1
    return m


# the general kernel's np; the fused kernel's with one p sign a lane and with two (shifted); the wide rows
# (np 128, 256), the q-window kernel (mixed, np 128), three states, the nonlinear coupling
TOL = {"fp64": 1e-12, "mixed": 2e-5}  # one right-hand side, as elsewhere
KINDS = [("two", 16), ("two", 32), ("shifted", 64), ("three", 64), ("one", 128), ("two", 128), ("two", 256), ("nonlinear", 32)]


CASES = [(k, n, p, "1") for k, n in KINDS for p in TOL] + [(k, 128, "mixed", "0") for k in ("one", "two")]


@pytest.mark.parametrize("nq", [1, 2, 3])
@pytest.mark.parametrize("kind,n_p,precision,window", CASES)
def test_rhs(nq, kind, n_p, precision, window, monkeypatch):
    monkeypatch.setenv("QHFPE_FUSED_WINDOW", window)
    m = _model(kind, nq, n_p)
    P = _P(m, precision)
    P.set_state(qi.random_state(m, seed=50 + nq))
    W = P.get_state(0)
    got = P.apply_rhs(0)
    P.close()
    assert rel(got, oracle.Oracle(m).rhs(W)) < TOL[precision]


def _steps(Ps, run, tol):
    W = []
    for k, P in enumerate(Ps):
        P.set_state(qi.random_state(P.model, seed=60 + k, hermitian=True))
        W.append(P.get_state(0))
    run()
    for P, w in zip(Ps, W):
        assert rel(P.get_state(0), oracle.Oracle(P.model).step(w, 3)[0]) < tol
        P.close()


@pytest.mark.parametrize("nq", [1, 2, 3])
@pytest.mark.parametrize("n_p", [32, 64])
def test_resident_steps(nq, n_p):
    P = _P(_model("two", nq, n_p), "mixed")
    _steps([P], lambda: P.step(3), 1e-5)


@pytest.mark.parametrize("precision,tol", [("mixed", 1e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("n_p", [32, 64])
def test_batch_with_one_row_a_block(n_p, precision, tol):
    """Members of 1 to 16 q rows beside one of 17: clusters of blocks with one row each."""
    from paper_1706_09590_gb300 import Batch
    ms = [_model("two", nq, n_p) for nq in (17, 16, 7, 3, 2, 1)]
    ms[2]["periodic_q"] = 0
    Ps = [_P(m, precision) for m in ms]
    B = Batch(Ps)
    _steps(Ps, lambda: (B.step(3), B.close()), tol)
