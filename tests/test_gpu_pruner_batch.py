"""Gradients of large batches (weight-gradient products cut along K, column sums in
slices) against the FP64 reference; the tolerances are those of the small batch
(BF16 operand rounding over the layer depths, which does not grow with the batch)."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F,H,B", [
    (65, 256, 4096),     # K of exactly 64 chunks
    (65, 200, 4111),     # ragged batch, H no multiple of 16
    (9, 32, 9001),       # one tile
    (65, 64, 20_000),
    (300, 300, 5000),    # several column tiles
])
def test_large_batch_gradients(F, H, B):
    import paper_2504_13446_gb300 as rkr
    p = mlp.init_params(F, H, 2)
    flat = mlp.flatten(p).astype(np.float32)
    p32 = mlp.unflatten(flat.astype(np.float64), F, H)
    rng = np.random.default_rng(B)
    X = (rng.standard_normal((B, F)) / np.sqrt(F)).astype(np.float32)
    t = rng.standard_normal(B).astype(np.float32)
    target = (3.0 - t + rng.standard_normal(B)).astype(np.float32)
    net = rkr.Pruner(F, H)
    net.set_params(flat)
    loss, g = net.loss_grads(X, t, target)
    loss_ref, g_ref = mlp.loss_and_grads(p32, X.astype(np.float64), t.astype(np.float64), target)
    assert abs(loss - loss_ref) <= 3e-2 * (1 + loss_ref)
    gf = mlp.unflatten(g.astype(np.float64), F, H)
    for k in mlp.ORDER:
        a, b = np.asarray(gf[k]).ravel(), np.asarray(g_ref[k]).ravel()
        assert np.linalg.norm(a - b) < 5e-2 * max(np.linalg.norm(b), 1e-12), k
    loss2, g2 = net.loss_grads(X, t, target)
    assert loss2 == loss and np.array_equal(g2, g)      # fixed order of summation
