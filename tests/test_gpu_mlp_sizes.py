"""GPU: loss and gradient of the FP32 network at minibatch sizes around its tiles (64 rows), the
parts of its sums over the samples (64) and the splits of its weight gradients (128 samples, a
multiple of 32), against the FP64 CPU network; bars as at 96 samples (loss 1e-5, gradient 1e-4:
FP32 activations, products accurate to FP32).

The reference is taken at the FP32 values of parameters and features, which is what the network
is given: the gradient jumps where a unit changes sides, and at 65 and 2433 rows one third-layer
unit lies within 2e-8 of zero and changes sides between the FP64 inputs and their FP32 values, so
that the FP64 network itself differs by 1.0e-2 and 1.0e-4 between the two."""
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
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    loss_ref, g_ref = mlp.loss_and_grad(f32(theta), f32(X), T)
    d = P.DMRG(make_problem("p", 2, 2, 0, seed=12))
    loss, g = d.mlp_loss_grad(theta, X, T, precision=P.MIXED_FP32)
    assert abs(loss - loss_ref) <= 1e-5 * abs(loss_ref)
    assert np.linalg.norm(g - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
    d.close()
