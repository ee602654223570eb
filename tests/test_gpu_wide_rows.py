"""The general stage kernel's rows of 128 and 256 p values (a warp a row, 32-byte accesses at 256, neighbours three at a
time) against the FP64 form: one to three states, ragged and single-row tiles, periodic q, the terminator, elements with no
neighbour, one, and more than two batches of three."""
import numpy as np
import pytest

import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu


def _models():
    per = qi.photoisomerization_two_state(nq=13, n_p=256, depth=2, n_matsubara=1)
    per["periodic_q"] = 1
    return {"one_state": qi.single_state(lambda q: 0.5 * q * q, nq=21, n_p=256, pr=(-16.0, 16.0), depth=0, dt=0.002),
            "two_states": qi.photoisomerization_two_state(nq=8, n_p=256, depth=5, n_matsubara=4),
            "three_states": qi.three_state(nq=9, n_p=256, depth=4),
            "three_states_128": qi.three_state(nq=11, n_p=128, depth=5),
            "two_states_128": qi.photoisomerization_two_state(nq=10, n_p=128, depth=4, n_matsubara=2), "periodic": per,
            "terminator": qi.harmonic_two_state(nq=10, n_p=256, pr=(-16.0, 16.0), depth=3, dt=0.002)}


@pytest.mark.parametrize("name", ["one_state", "two_states", "three_states", "three_states_128", "two_states_128",
                                  "periodic", "terminator"])
@pytest.mark.parametrize("tile", ["1", "3"])
def test_rows(name, tile, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1706_09590_gb300 import Propagator
    monkeypatch.setenv("QHFPE_TILE_ROWS", tile)
    monkeypatch.setenv("QHFPE_FUSED_WINDOW", "0")
    m = _models()[name]
    W = qi.random_state(m, seed=5).astype(np.complex64).astype(np.complex128)
    L = {}
    for prec in ("mixed", "fp64"):
        P = Propagator(m, qi.u_table(m), precision=prec)
        P.set_state(W)
        L[prec] = P.apply_rhs(0, 31)
        P.close()
    # FP32 sums of at most 40 roundings, the terms together up to twice the result (the q stencil's weights), inputs
    # exact: 80 x 2^-24 = 4.8e-6 of the norm
    assert np.linalg.norm(L["mixed"] - L["fp64"]) < 4.8e-6 * np.linalg.norm(L["fp64"])
