"""GPU: loss and gradient of the FP32 network at minibatch sizes around its tiles (64 rows), the
parts of its sums over the samples (64) and the splits of its weight gradients (128 samples, a
multiple of 32), against the FP64 CPU network; bars as at 96 samples (loss 1e-5, gradient 1e-4:
FP32 activations, products accurate to FP32)."""
import numpy as np
import pytest

from gen import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 31, 64, 65, 127, 129, 255, 2433])
def test_gradient_at_tile_edges(rows):
    from paper_1507_00161_gb300.build import build
    build()
    import paper_1507_00161_gb300 as P
    from oracle import mlp
    rng = np.random.default_rng(100 + rows)
    theta = rng.standard_normal(mlp.n_params()) * 0.1
    X = rng.standard_normal((rows, 4))
    T = rng.standard_normal(rows)
    loss_ref, g_ref = mlp.loss_and_grad(theta, X, T)
    d = P.DMRG(make_problem("p", 2, 2, 0, seed=12))
    loss, g = d.mlp_loss_grad(theta, X, T, precision=P.MIXED_FP32)
    assert abs(loss - loss_ref) <= 1e-5 * abs(loss_ref)
    assert np.linalg.norm(g - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
    d.close()
