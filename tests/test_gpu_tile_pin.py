"""QHFPE_TILE_ROWS: a height of the stage kernel pins that kernel and its tile; a value that is no height changes nothing."""
import pytest

import qhfpe_inputs as qi

pytestmark = pytest.mark.gpu


def _tile(monkeypatch, value, n=1):
    from paper_1706_09590_gb300 import Batch, Propagator
    if value is None:
        monkeypatch.delenv("QHFPE_TILE_ROWS", raising=False)
    else:
        monkeypatch.setenv("QHFPE_TILE_ROWS", value)
    Ps = []
    for k in range(n):
        m = qi.harmonic_two_state(nq=24 + k, depth=2)
        Ps.append(Propagator(m, qi.u_table(m), precision="mixed"))
        Ps[-1].set_state(qi.random_state(m, seed=k))
    if n == 1:
        Ps[0].step(2)
        t = Ps[0].tile_rows()
    else:
        B = Batch(Ps)
        B.step(2)
        t = B.tile_rows()
        B.close()
    for P in Ps:
        P.close()
    return t


@pytest.mark.parametrize("n", [1, 2])
def test_pin(n, monkeypatch):
    assert _tile(monkeypatch, None, n) == 0  # cluster-resident
    for no_height in ("", "0", "-3", "99999", "auto"):
        assert _tile(monkeypatch, no_height, n) == 0
    assert _tile(monkeypatch, "3", n) == 3
