"""The training kernels of the warm-start network at the edges of their tiles
(32 columns, 16 or 32 rows, 16x16 in the weight gradient), rows that are not
16-byte aligned, and gradients that add up over backward passes."""
import numpy as np
import pytest

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [(1, 1, 1), (1, 3, 40), (2, 16, 32), (1, 17, 33), (1, 31, 30), (1, 33, 64), (3, 15, 17), (1, 70, 5)]


@pytest.mark.parametrize("c", [6, 10])
@pytest.mark.parametrize("shape", SHAPES)
def test_forward_and_gradients(c, shape):
    from paper_1109_1146_gb300.mf import CNN
    N, H, W = shape
    rng = np.random.Generator(np.random.PCG64(N * 10007 + H * 101 + W + c))
    net = CNN(channels=c, seed=5)
    p = net.get_params()
    x = rng.standard_normal((N, c, H, W)).astype(np.float32)
    dy = rng.standard_normal((N, c, H, W)).astype(np.float32)
    xt, dyt = torch.from_numpy(x).cuda(), torch.from_numpy(dy).cuda()
    yt = torch.empty_like(xt)
    net.forward(xt, yt)
    ref, _, _ = ocnn.forward(p, x.astype(np.float64), c)
    # sums of at most 288 products of O(1) terms over four layers, 2^-24 each
    np.testing.assert_allclose(yt.cpu().numpy(), ref, rtol=1e-4, atol=1e-4)
    net.zero_grad()
    net.backward(xt, dyt)
    g = net.get_grads()
    gref = ocnn.backward(p, x.astype(np.float64), c, dy.astype(np.float64))
    scale = float(np.abs(gref).max())
    np.testing.assert_allclose(g, gref, rtol=2e-3, atol=2e-4 * scale)
    # a second pass adds the same gradients, bit for bit (no atomics)
    net.backward(xt, dyt)
    np.testing.assert_array_equal(net.get_grads(), g + g)
