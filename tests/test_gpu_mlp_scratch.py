"""The scratch of the network's backward pass grows with the corpora that a model sees: gradients of larger and smaller
ones in turn are those of a model that sees each alone, bit for bit."""
import numpy as np
import pytest

import paper_1411_4212_gb300 as rw

pytestmark = pytest.mark.gpu

SHIFT = np.array([-1.9, 0.19, 1.0, 0.4, 0.0, 0.0], dtype=np.float32)
SCALE = np.array([1 / 1.1, 20.0, 1.0, 5.0, 10.0, 1.0], dtype=np.float32)


def _gradient(net, n):
    x = np.zeros((n, 6), dtype=np.float32)
    x[:, 0] = np.linspace(-3.3, -0.01, n)
    x[:, 1], x[:, 2], x[:, 3] = 0.2, 1.0, 0.45
    t = (-0.3 * x[:, 0] ** 2).astype(np.float32)
    return net.gradient(x, t, np.array([0, n], dtype=np.int32))


def test_corpora_of_different_sizes_through_one_model():
    net = rw.Mlp(SHIFT, SCALE, seed=3)
    for n in (1, 33, 17, 2000, 1999, 45000, 16):
        alone = rw.Mlp(SHIFT, SCALE, seed=3)
        L0, g0 = _gradient(alone, n)
        L1, g1 = _gradient(net, n)
        assert L0 == L1 and np.array_equal(g0.view(np.int32), g1.view(np.int32)), n
        alone.close()
    net.close()
