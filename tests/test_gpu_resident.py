"""Cluster-resident propagation (small two-state propagators, mixed form) against the launch-per-stage form:
ragged row counts, every cluster size that the replica counts lead to, periodic q, closures, and runs
longer than one launch."""
import numpy as np
import pytest

import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu

# two FP32 evaluations that differ in rounding order: 6e-8 a stage, over some tens of steps
TOL = 3e-6


def _run(m, reps, steps, resident, monkeypatch):
    from paper_1706_09590_gb300 import Propagator
    monkeypatch.setenv("QHFPE_RESIDENT", "1" if resident else "0")
    P = Propagator(m, qi.u_table(m), precision="mixed", n_replicas=reps)
    for r in range(reps):
        P.set_state(qi.random_state(m, seed=40 + r % 5, hermitian=True), r)
    tr = [P.step(steps, record_trace=True)]
    P.step(2)  # without traces
    tr.append(P.step(3, record_trace=True))
    assert (P.tile_rows() == 0) == resident  # the stage kernel's tile is not chosen when nothing launches it
    out = [P.get_state(r) for r in sorted({0, reps // 2, reps - 1})]
    P.close()
    return out, tr


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


def _compare(m, reps, steps, monkeypatch):
    (a, ta), (b, tb) = _run(m, reps, steps, True, monkeypatch), _run(m, reps, steps, False, monkeypatch)
    for x, y in zip(a + ta, b + tb):
        assert rel(x, y) < TOL, rel(x, y)


@pytest.mark.parametrize("n_p", [32, 64])
@pytest.mark.parametrize("nq,reps", [(5, 1), (17, 1), (32, 3), (33, 20), (19, 90)])
def test_resident_row_counts_and_cluster_sizes(n_p, nq, reps, monkeypatch):
    _compare(qi.harmonic_two_state(nq=nq, n_p=n_p, depth=2, dt=0.004), reps, 10, monkeypatch)


@pytest.mark.parametrize("name", ["periodic", "truncated", "matsubara", "one_element"])
def test_resident_models(name, monkeypatch):
    m = {"periodic": qi.harmonic_two_state(nq=18, depth=3, periodic_q=1),
         "truncated": qi.harmonic_two_state(nq=21, depth=5, closure=0),
         "matsubara": qi.photoisomerization_two_state(nq=24, n_p=32, depth=2, n_matsubara=2, dt=2e-3),
         "one_element": qi.harmonic_two_state(nq=20, depth=0)}[name]
    _compare(m, 2, 12, monkeypatch)


def test_resident_longer_than_one_launch(monkeypatch):
    _compare(qi.harmonic_two_state(nq=6, depth=0, dt=1e-5), 1, 4100, monkeypatch)


def test_resident_is_left_out_where_it_does_not_fit(monkeypatch):
    """A state beyond a cluster's shared memory keeps the launch-per-stage form."""
    from paper_1706_09590_gb300 import Propagator
    monkeypatch.setenv("QHFPE_RESIDENT", "1")
    m = qi.photoisomerization_two_state(nq=60, n_p=64, depth=6, n_matsubara=2)
    P = Propagator(m, qi.u_table(m), precision="mixed")
    P.set_state(qi.random_state(m, seed=1))
    P.step(1)
    assert P.tile_rows() > 0
    P.close()
