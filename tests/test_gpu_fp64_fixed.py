"""The FP64 stage kernel's integer arithmetic where it can go wrong: every np and state count against the oracle,
rows of very different and extreme magnitudes, non-finite values, and the shapes that keep FP64 sums (many
tier neighbours, a p axis on which a lane holds both signs)."""
import numpy as np
import pytest

import oracle
import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu

# FP64: a sum of some tens of terms, each rounded at 1.1e-16 of values up to a hundred times the result
TOL = 2e-14


def _P(m):
    from paper_1706_09590_gb300 import Propagator
    return Propagator(m, qi.u_table(m), precision="fp64")


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


def _models():
    out = {}
    for n_p in (32, 64, 128, 256):
        out[f"two_{n_p}"] = qi.photoisomerization_two_state(nq=11, n_p=n_p, depth=2, n_matsubara=1)
    out["three_64"] = qi.three_state(nq=7, n_p=64, depth=1, n_matsubara=1)
    out["three_256"] = qi.three_state(nq=5, n_p=256, depth=1, n_matsubara=0)
    out["one_128"] = qi.single_state(lambda q: 0.5 * q * q, nq=18, n_p=128, depth=3)
    per = qi.harmonic_two_state(nq=9, n_p=64, depth=2, periodic_q=1)
    out["periodic_terminator"] = per
    # p = 0 inside a lane's run of values, and 13 tier neighbours: the sums in FP64
    out["shifted_p"] = qi.harmonic_two_state(nq=9, n_p=128, pr=(-8.3, 7.7), depth=2)
    out["many_neighbours"] = dict(qi.single_state(lambda q: 0.5 * q * q, nq=4, n_p=32, depth=6, closure=0),
                                  n_matsubara=6, high_temperature=0, use_cdelta=1, beta=1.0)
    return out


MODELS = _models()


@pytest.mark.parametrize("name", list(MODELS))
def test_rhs_against_oracle(name):
    m = MODELS[name]
    W = qi.random_state(m, seed=31)
    P = _P(m)
    P.set_state(W)
    got = P.apply_rhs(0)
    P.close()
    assert rel(got, oracle.Oracle(m).rhs(W)) < TOL


@pytest.mark.parametrize("scale", [1e-200, 1e200])
def test_extreme_magnitudes(scale):
    """The right-hand side is linear: scaled inputs give scaled outputs, also with rows far apart."""
    m = MODELS["two_128"]
    W = qi.random_state(m, seed=32) * 10.0 ** np.linspace(-40, 40, m["nq"])[:, None]
    P = _P(m)
    out = []
    for s in (1.0, scale):
        P.set_state(W * s)
        out.append(P.apply_rhs(0) / s)
    ref = oracle.Oracle(m).rhs(W)
    P.close()
    for i in range(m["nq"]):  # row by row: each has its own magnitude
        assert rel(out[0][..., i, :], ref[..., i, :]) < TOL
        assert rel(out[1][..., i, :], out[0][..., i, :]) < TOL


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_stay_visible(bad):
    from paper_1706_09590_gb300 import QhfpeError
    m = MODELS["two_64"]
    W = qi.random_state(m, seed=33)
    W[0, 1, 0, 5, 17] = bad
    P = _P(m)
    with pytest.raises(QhfpeError):
        P.set_state(W)  # reported; the replica holds the value
    got = P.apply_rhs(0)
    P.close()
    assert not np.isfinite(got[0, 1, 0, 5]).any()  # its transform
    far = [e for e in range(got.shape[0]) if e != 0]
    assert np.isfinite(got[0][:, :, 9:]).all() and np.isfinite(got[far][:, :, :, :5]).all()  # rows it does not reach
