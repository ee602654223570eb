"""The q-window stage kernel with the potential term from the tensor-core kernel, against the general stage
kernel on the same term: ragged tiles, periodic q, one state, the terminator and the delta-term."""
import numpy as np
import pytest

import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu


def _models():
    per = qi.photoisomerization_two_state(nq=25, n_p=128, depth=2, n_matsubara=1)
    per["periodic_q"] = 1
    return {"ragged": qi.photoisomerization_two_state(nq=7, n_p=128, depth=3, n_matsubara=2), "periodic": per,
            "terminator": qi.harmonic_two_state(nq=30, n_p=128, pr=(-16.0, 16.0), depth=3, dt=0.002),
            "one_state": qi.single_state(lambda q: 0.5 * q * q, nq=37, n_p=128, pr=(-16.0, 16.0), depth=3, dt=0.002)}


@pytest.mark.parametrize("name", ["ragged", "periodic", "terminator", "one_state"])
def test_window_with_external_potential(name, monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1706_09590_gb300 import Propagator
    m = _models()[name]
    W = qi.random_state(m, seed=9)
    monkeypatch.setenv("QHFPE_TILE_ROWS", "2")
    out = {}
    for flag in ("1", "0"):
        monkeypatch.setenv("QHFPE_FUSED_WINDOW", flag)
        P = Propagator(m, qi.u_table(m), precision="bf16x3")
        P.set_state(W)
        P.step(3)
        assert P.stage_form() == int(flag)
        out[flag] = P.get_state(0)
        P.close()
    # one potential term, FP32 sums in another order; the bf16 split of inputs that differ in their last bit
    # differs by 2^-24 of them
    assert np.linalg.norm(out["1"] - out["0"]) < 3e-6 * np.linalg.norm(out["0"])
