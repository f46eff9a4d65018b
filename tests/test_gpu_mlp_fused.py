"""The fused network kernels (all layers of a row block in one launch, all
layers' gradients in another) at the shapes where they can go wrong: widths
that are no multiple of four, one row, one row more than a block, row counts
at the changes of the block height, and a network too wide for shared memory
(the layer-by-layer kernels).

Tolerances as in test_gpu_mlp.py (FP32 sums against FP64: 1e-4 of the largest
value), and the loss of a training step must equal loss_grad's on the same
parameters bit for bit (same kernels' arithmetic).
"""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[5, 128, 128, 128, 64], [3, 17, 9], [1, 1, 1], [6, 33, 33, 7], [5, 300, 300, 12]])
@pytest.mark.parametrize("n", [1, 3, 65, 305, 611])
def test_shapes(lbm, sizes, n):
    rng = np.random.default_rng(n)
    net = lbm.WarmStartNet(sizes[0], sizes[1], len(sizes) - 2, sizes[-1])
    theta = rng.normal(0, 0.1, net.n_params).astype(np.float32)
    net.set_params(theta)
    X = rng.uniform(-1, 1, (n, sizes[0])).astype(np.float32)
    Y = rng.normal(0, 1, (n, sizes[-1])).astype(np.float32)
    sc = [rng.normal(0, 0.1, sizes[0]), rng.uniform(0.5, 2, sizes[0]), rng.normal(0, 0.1, sizes[-1]), rng.uniform(0.5, 2, sizes[-1])]
    sc = [v.astype(np.float32) for v in sc]
    net.set_scaling(*sc)
    sd = [v.astype(np.float64) for v in sc]
    loss, g = net.loss_grad(X, Y)
    ref_loss, ref_g = mlp.loss_and_grad(theta.astype(np.float64), sizes, X, Y, *sd)
    assert loss == pytest.approx(ref_loss, rel=1e-4)
    assert np.abs(g - ref_g).max() < 1e-4 * np.abs(ref_g).max()
    out = net.predict(X)
    ref, _ = mlp.forward(theta.astype(np.float64), sizes, X, sd[0], sd[1])
    want = ref * sd[3] + sd[2]
    assert np.abs(out - want).max() < 1e-4 * np.abs(want).max()
    # Adam over minibatches that do not divide the set, then the loss at the end
    final = net.train(X, Y, epochs=3, batch=17, lr=1e-3, seed=3)
    again, _ = net.loss_grad(X, Y)
    assert final == again
    net.close()
