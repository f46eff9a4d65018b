"""Training against its own definition, bit for bit: every epoch is one
minibatch (the whole set in that epoch's order), its gradient is loss_grad's of
the same rows at the same parameters, and Adam is
    m1 <- fma(1 - b1, g, b1 m1),  m2 <- fma((1 - b2) g, g, b2 m2),
    p  <- p - lr (m1 / c1) / (sqrt(m2 / c2) + eps)
in FP32 with IEEE division and root.  A fused multiply-add of floats is their
FP64 product (exact) and sum, rounded to FP32.  Both kernels that apply it (the
fused gradients, and the layered path of networks too wide for shared memory)
must agree."""
import ctypes
import ctypes.util

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
F = np.float32
M64 = (1 << 64) - 1


def splitmix(x):
    z = (x + 0x9E3779B97F4A7C15) & M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def order(n, epoch, seed):
    """The epoch's Fisher-Yates order of n rows."""
    perm = list(range(n))
    for i in range(n - 1, 0, -1):
        j = splitmix(seed ^ (epoch << 32) ^ i) % (i + 1)
        perm[i], perm[j] = perm[j], perm[i]
    return np.array(perm)


def fma(a, b, c):
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(F)


@pytest.mark.parametrize("sizes", [(5, 128, 3, 64), (3, 17, 2, 9), (5, 300, 2, 12)])
def test_training_is_its_definition(lbm, sizes):
    powf = ctypes.CDLL(ctypes.util.find_library("m")).powf
    powf.restype, powf.argtypes = ctypes.c_float, [ctypes.c_float, ctypes.c_float]
    n, epochs, seed, lr = 40, 6, 11, F(1e-3)
    rng = np.random.default_rng(1)
    X = rng.uniform(-1, 1, (n, sizes[0])).astype(F)
    Y = rng.normal(0, 1, (n, sizes[-1])).astype(F)
    net, ref = (lbm.WarmStartNet(*sizes, seed=4) for _ in range(2))
    p = net.get_params()
    m1, m2 = np.zeros_like(p), np.zeros_like(p)
    b1, b2, eps = F(0.9), F(0.999), F(1e-8)
    for ep in range(epochs):
        ref.set_params(p)
        perm = order(n, ep, seed)
        _, g = ref.loss_grad(X[perm], Y[perm])
        m1 = fma(F(1) - b1, g, b1 * m1)
        m2 = fma((F(1) - b2) * g, g, b2 * m2)
        c1, c2 = (F(1) - F(powf(b, F(ep + 1))) for b in (b1, b2))
        p = p - lr * (m1 / c1) / (np.sqrt(m2 / c2) + eps)
    net.train(X, Y, epochs, batch=n, lr=float(lr), seed=seed)
    got = net.get_params()
    net.close()
    ref.close()
    assert np.array_equal(got, p), int((got != p).sum())
