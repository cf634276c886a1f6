"""The sums of the predictor's gradient over the cells: the same bits on every call,
and no further from 64 bits than sums of 1024 cells in a row.

The bound: on these inputs, with operands rounded to FP32 and exact otherwise, the
weight gradients are off by 1.25e-7 to 2.1e-7 of their norm where 1024 cells are added
in a row and the rows' sums one after another, by 2.2e-7 to 2.4e-7 where 256 are, and
by 4.5e-8 to 5.5e-8 as chains of 64 cells added as a tree (computed on the host, the
three seeds).  The gradient also carries the rounding of its operands' own sums, of
144 terms a layer; the least of the first order, 1.25e-7, leaves room for it.
"""
import numpy as np
import pytest

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


def inputs(seed, n, h, w):
    """Smooth planes as a regrid makes them, targets and mask."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:h, 0:w] / 64.0
    f = np.zeros((n, ocnn.C_IN, h, w))
    for k in range(n):
        p = rng.uniform(0, 6.28, 4)
        wave = np.sin(2.1 * x + p[0]) * np.cos(1.7 * y + p[1]) + 0.5 * np.sin(5.3 * (x - y) + p[2])
        f[k, 0], f[k, 1] = 1.5 * wave, np.clip(2.0 + 2.0 * np.sin(0.7 * x + p[3]), -1, 5)
        f[k, 2], f[k, 3] = np.abs(3.0 * np.cos(2.3 * x + p[1])), np.abs(2.0 * np.cos(1.9 * y + p[2]))
        f[k, 4] = np.abs(wave) > 0.8
    t = np.maximum(f[:, 4], np.roll(f[:, 4], 2, axis=2))
    m = np.ones((n, h, w))
    m[:, : h // 8] = 0.0
    theta = ocnn.init_params(seed).astype(np.float32).astype(np.float64)
    return theta, f.astype(np.float32).astype(np.float64), t, m


# one tile; several tiles of a few CTAs; 320 and 640 tiles on 304 CTAs, of which some take two and three
@pytest.mark.parametrize("n,h,w", [(1, 8, 32), (2, 9, 65), (5, 128, 128), (40, 64, 64)])
def test_gradient_has_the_same_bits_on_every_call(n, h, w):
    from paper_1901_06798_gb300 import binding
    a = inputs(n, n, h, w)
    loss, g = binding.cnn_loss_grad(*a)
    for _ in range(4):
        loss2, g2 = binding.cnn_loss_grad(*a)
        assert loss2 == loss and np.array_equal(g2, g)
    loss_ref, g_ref = ocnn.backward(*a)
    assert loss == pytest.approx(loss_ref, rel=1e-5)
    assert np.abs(g - g_ref).max() <= 1e-4 * np.abs(g_ref).max()


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_gradient_error_of_the_sums(seed):
    from paper_1901_06798_gb300 import binding
    a = inputs(seed, 4, 128, 128)
    _, g = binding.cnn_loss_grad(*a)
    _, ref = ocnn.backward(*a)
    err = np.linalg.norm(np.asarray(g, dtype=np.float64) - ref) / np.linalg.norm(ref)
    print(f"gradient off by {err:.2e} of its norm")
    assert err <= 1.25e-7
