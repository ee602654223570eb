"""The FP64 form's results do not depend on the tile that the autotuner picks: states after a few steps and traces are equal
bit for bit over tile heights, also where rows of one tile are of very different magnitude."""
import numpy as np
import pytest

import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu


def _models():
    return {"two_128": qi.photoisomerization_two_state(nq=21, n_p=128, depth=2, n_matsubara=1),
            "two_32": qi.harmonic_two_state(nq=18, n_p=32, depth=3),
            "periodic_64": qi.harmonic_two_state(nq=19, n_p=64, depth=2, periodic_q=1),
            "three_64": qi.three_state(nq=13, n_p=64, depth=1, n_matsubara=1),
            "one_256": qi.single_state(lambda q: 0.5 * q * q, nq=11, n_p=256, pr=(-16.0, 16.0), depth=2, dt=1e-3),
            # groups of three rows: between two and three rows of elements for each block of a wave
            "one_128_threes": qi.single_state(lambda q: 0.5 * q * q, nq=101, n_p=128, pr=(-16.0, 16.0), depth=14, dt=1e-4),
            "two_128_threes": qi.photoisomerization_two_state(nq=62, n_p=128, depth=3)}


@pytest.mark.parametrize("name", list(_models()))
@pytest.mark.parametrize("steep", [False, True])
def test_states_are_equal_over_tile_heights(name, steep, monkeypatch):
    from paper_1706_09590_gb300 import Propagator
    m = _models()[name]
    W = qi.random_state(m, seed=71, hermitian=True)
    if steep:  # from row to row
        W *= 10.0 ** (-3.0 * (np.arange(m["nq"]) % 5))[:, None]
    out = []
    for tile in (1, 2, 3, 4, 6):
        monkeypatch.setenv("QHFPE_TILE_ROWS", str(tile))
        P = Propagator(m, qi.u_table(m), precision="fp64")
        P.set_state(W)
        tr = P.step(3, record_trace=True)
        out.append((P.get_state(0), tr, P.tile_rows()))
        P.close()
    assert len({t for _, _, t in out}) > 1
    for a, tr, _ in out[1:]:
        assert np.array_equal(a, out[0][0]) and np.array_equal(tr, out[0][1])
