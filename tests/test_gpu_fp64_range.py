"""The FP64 form over the whole range of doubles: the right-hand side is linear, so states scaled by a power of two give
the scaled result (to the spacing of subnormal numbers), and infinities stay where the sums of doubles have them."""
import numpy as np
import pytest

import oracle
import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu

TOL = 2e-14  # FP64 sums of some tens of terms, as elsewhere
TINY = 2.0 ** -1074


def _models():
    nl = qi.harmonic_two_state(nq=9, n_p=32, depth=2, closure=0)
    nl["v_c2"] = 0.1
    return {"two_128": qi.photoisomerization_two_state(nq=11, n_p=128, depth=2, n_matsubara=1),
            "two_32": qi.harmonic_two_state(nq=13, n_p=32, depth=3),
            "three_64": qi.three_state(nq=7, n_p=64, depth=1, n_matsubara=1),
            "one_256": qi.single_state(lambda q: 0.5 * q * q, nq=6, n_p=256, pr=(-16.0, 16.0), depth=2),
            "shifted_p": qi.harmonic_two_state(nq=9, n_p=64, pr=(-7.75, 8.25), depth=2), "nonlinear": nl}


MODELS = _models()


def _P(m):
    from paper_1706_09590_gb300 import Propagator
    return Propagator(m, qi.u_table(m), precision="fp64")


def _rhs(P, W):
    P.set_state(W)
    return P.apply_rhs(0)


def _rows(a):
    return np.linalg.norm(a, axis=-1)


@pytest.mark.parametrize("name", list(MODELS))
@pytest.mark.parametrize("k", [-1060, -1020, -960, -890, 900, 1000, 1010])
def test_scaled_states(name, k):
    """2^1010: inputs from 2^1007 on, results (rates up to some hundreds) below 2^1024."""
    m = MODELS[name]
    W = qi.random_state(m, seed=91)
    h = k // 2
    Ws = W * 2.0 ** h * 2.0 ** (k - h)
    P = _P(m)
    ref = _rhs(P, Ws * 2.0 ** -h * 2.0 ** (h - k))  # (of the values that are left in subnormal numbers)
    got = _rhs(P, Ws)
    P.close()
    assert np.isfinite(got).all()
    err = np.abs((got * 2.0 ** -h) * 2.0 ** (h - k) - ref)
    # sums of terms rounded at the spacing of subnormal numbers: some tens of them, weighted by rates
    rate = np.linalg.norm(ref) / np.linalg.norm(W)
    slack = 64 * (1 + rate) * 2.0 ** (-1074 - k) if k < -900 else 0.0
    assert (err <= TOL * _rows(ref)[..., None] * 16 + slack).all()


@pytest.mark.parametrize("name", ["two_128", "two_32", "nonlinear"])
def test_rows_far_apart(name):
    """Rows from the subnormal range to 1e300 in one state, beside each other: each row against the oracle."""
    m = MODELS[name]
    nq = m["nq"]
    W = qi.random_state(m, seed=92) * 10.0 ** np.where(np.arange(nq) % 3 == 0, -309.0, np.where(np.arange(nq) % 3 == 1, -280.0, 300.0))[:, None]
    W[..., nq // 2:, :] = 0.0  # and rows of zeros
    W[..., -1, :] = 1e-300
    P = _P(m)
    got = _rhs(P, W)
    P.close()
    ref = oracle.Oracle(m).rhs(W)
    a, b = _rows((got - ref) * 2.0 ** -600), _rows(ref * 2.0 ** -600)  # (norms within the range of doubles)
    assert (a <= TOL * b + 1e-300).all()
    small = np.abs(ref).max(axis=-1) < 1e-200  # rows without large neighbours
    assert (np.abs(got - ref).max(axis=-1)[small] <= 1e-12 * np.abs(ref).max(axis=-1)[small] + 1e6 * TINY).all()


def test_zero_state_gives_zero():
    m = MODELS["two_128"]
    P = _P(m)
    W = np.zeros_like(qi.random_state(m))
    W[..., ::2] *= -1.0  # both zeros
    assert not _rhs(P, W).any()
    P.close()


@pytest.mark.parametrize("name", ["two_128", "two_32"])
def test_an_infinity_reaches_what_it_reaches(name):
    """One infinite value: its row (by the transform), its column within the q stencil, and its p neighbours in the elements
    coupled to it are not finite; everything else is what it is without it."""
    from paper_1706_09590_gb300 import QhfpeError
    m = MODELS[name]
    W = qi.random_state(m, seed=93)
    P = _P(m)
    clean = _rhs(P, W)
    W[0, 1, 0, 4, 9] = np.inf
    with pytest.raises(QhfpeError):
        P.set_state(W)  # reported; the replica holds it
    got = P.apply_rhs(0)
    P.close()
    p = m["p_min"] + 9 * (m["p_max"] - m["p_min"]) / m["np"]
    hit = np.zeros(got.shape, dtype=bool)
    hit[0, :, :, 4] = True
    reach = range(-2, 4) if p >= 0 else range(-3, 3)  # rows whose upwind difference reads row 4
    for d in reach:
        hit[0, 1, 0, 4 + d, 9] = True
    hit[1:, 1, 0, 4, 7:12] = True  # elements coupled to element 0 (or not)
    # (not bit for bit: where a column's values are far apart its neighbours' sums are taken at another unit)
    assert np.linalg.norm(got[~hit] - clean[~hit]) < TOL * np.linalg.norm(clean[~hit])
    assert not np.isfinite(got[0, 1, 0, 4]).any() and not np.isfinite(got[0, 1, 0, [4 + d for d in reach], 9]).any()


@pytest.mark.parametrize("k", [-850, 900, 990, 1006])
def test_large_rates(k):
    """Fast q differences (p / 60 dq up to 2^20) of values near the ends: finite results, infinities where they overflow."""
    m = qi.harmonic_two_state(nq=9, n_p=32, qr=(-1e-5, 1e-5), pr=(-128.0, 128.0), depth=1, eta=0.0)
    W = qi.random_state(m, seed=94)
    h = k // 2
    P = _P(m)
    ref = _rhs(P, W)
    got = _rhs(P, W * 2.0 ** h * 2.0 ** (k - h))
    P.close()
    back = (got * 2.0 ** -h) * 2.0 ** (h - k)
    fits = np.abs(ref) < 2.0 ** min(1022 - k, 1000)
    assert (np.abs(back - ref)[fits] <= 16 * TOL * np.broadcast_to(_rows(ref)[..., None], ref.shape)[fits]).all()
    assert not np.isfinite(got[~(np.abs(ref) < 2.0 ** min(1025 - k, 1000))]).any()
