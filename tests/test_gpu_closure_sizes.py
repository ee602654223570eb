"""Gradients of both closure networks at the batch sizes where the tiled products and the batch slices of the
weight gradients can go wrong (one point, tile edges, an odd count, slices that come out empty)."""
import numpy as np
import pytest

from oracle import closure as ocl

pytestmark = pytest.mark.gpu

# FP32 sums of at most 256 terms through four layers: a few 1e-6 relative in 2-norm; 1e-4 leaves room for
# cancellation in the output residuals
TOL = 1e-4
SIZES = [1, 63, 65, 257, 2049, 4100]


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


@pytest.mark.parametrize("n", SIZES)
def test_coefficient_network_gradient(torch, n):
    from paper_1706_09590_gb300.qhfpe import closure_loss_grad
    rng = np.random.default_rng(n)
    w = ocl.init_weights(5)
    w[-ocl.N_OUT * (ocl.N_HID + 1):] = rng.normal(size=ocl.N_OUT * (ocl.N_HID + 1)) * 0.02
    w = w.astype(np.float32)
    X = rng.uniform(-1, 1, (n, 3))
    phi, y = rng.normal(size=(n, 12, 10)), rng.normal(size=(n, 12))
    a, b = np.triu_indices(10)
    G = np.einsum("nsa,nsb->nab", phi, phi)[:, a, b]
    stats = np.concatenate([G, np.einsum("nsa,ns->na", phi, y), (y * y).sum(1)[:, None], np.full((n, 1), 12.0)], axis=1)
    L_ref, g_ref = ocl.loss_and_grad(w.astype(np.float64), X, stats, 0.05)
    L, g = closure_loss_grad(w, X, stats, 0.05)
    assert L == pytest.approx(L_ref, rel=TOL)
    assert rel(g.astype(np.float64), g_ref) < TOL


@pytest.mark.parametrize("S,n", [(1, 65), (1, 257), (2, 1), (2, 2049)])
def test_state_network_gradient(torch, S, n):
    from paper_1706_09590_gb300.qhfpe import closure_state_loss_grad
    n_in, n_out = ocl.state_sizes(S)
    rng = np.random.default_rng(n)
    w = (rng.normal(size=ocl.state_n_weights(S)) * 0.05).astype(np.float32)
    w[-3:] = 1.0
    X = rng.normal(size=(n, n_in)).astype(np.float32)
    Y = rng.normal(size=(n, n_out)).astype(np.float32)
    L_ref, g_ref = ocl.state_loss_and_grad(w.astype(np.float64), X.astype(np.float64), Y.astype(np.float64), S)
    L, g = closure_state_loss_grad(S, w, X, Y)
    assert L == pytest.approx(L_ref, rel=TOL)
    assert rel(g.astype(np.float64), g_ref) < TOL
