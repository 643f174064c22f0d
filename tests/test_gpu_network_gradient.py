"""Loss and gradient of the initial-guess network (am_mlp_loss_grad) against
the same network in 64 bits, at the sample counts where the tiled kernels
change: one sample, the edges of the 32- and 64-row tiles, of the sample
chunks of the weight gradient and of the tile choice."""
import numpy as np
import pytest

from paper_2107_10800_gb300 import build, binding

pytestmark = pytest.mark.gpu

LAYERS = (144, 256, 256, 256, 32)
# FP32 sums of up to 256 products per layer and pass: about sqrt(256) 2^-24
# = 1e-6 of the result each, over four layers forward and four backward
TOL = 1e-5


@pytest.fixture(scope="module")
def net():
    build.build()
    m = binding.Mlp()
    rng = np.random.default_rng(5)
    flat = []
    for k, n in zip(LAYERS[:-1], LAYERS[1:]):
        flat += [rng.standard_normal(n * k) * np.sqrt(2.0 / k), 0.1 * rng.standard_normal(n)]
    m.set_params(np.concatenate(flat).astype(np.float32))
    yield m
    m.close()


def exact(p, X, T):
    """Loss, gradient, and per parameter block what the units whose input is
    so near zero that FP32 does not determine their ReLU mask can change:
    each such unit's mask is turned over by itself."""
    p, a, T = p.astype(np.float64), X.astype(np.float64), T.astype(np.float64)
    acts, pre, Ws, k = [a], [], [], 0
    for i, (n_in, n_out) in enumerate(zip(LAYERS[:-1], LAYERS[1:])):
        W = p[k:k + n_in * n_out].reshape(n_out, n_in)
        b = p[k + n_in * n_out:k + n_in * n_out + n_out]
        k += n_in * n_out + n_out
        z = a @ W.T + b
        a = np.maximum(z, 0.0) if i < 3 else z
        acts.append(a)
        pre.append(z)
        Ws.append(W)

    def gradient(flip=None):
        d, blocks = 2.0 * (a - T) / a.size, []
        for i in range(3, -1, -1):
            blocks = [d.T @ acts[i], d.sum(axis=0)] + blocks
            if i:
                mask = pre[i - 1] > 0
                if flip is not None and flip[0] == i - 1:
                    mask[flip[1:]] ^= True
                d = (d @ Ws[i]) * mask
        return blocks

    g = gradient()
    slack = np.zeros(len(g))
    for i in range(3):
        for r, o in zip(*np.nonzero(np.abs(pre[i]) < 1e-5)):
            slack += [np.linalg.norm(x - y) for x, y in zip(gradient((i, r, o)), g)]
    return ((a - T) ** 2).mean(), g, slack


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 65, 127, 256, 300, 608, 641, 1024, 1025, 2433])
def test_loss_and_gradient(net, n):
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, LAYERS[0])).astype(np.float32)
    T = rng.standard_normal((n, LAYERS[-1])).astype(np.float32)
    loss, grad = net.loss_grad(X, T)
    loss_x, blocks, slack = exact(net.params(), X, T)
    assert abs(loss - loss_x) <= TOL * loss_x
    off = 0
    for gx, sl in zip(blocks, slack):  # weights and biases layer by layer
        g = grad[off:off + gx.size].reshape(gx.shape)
        assert np.linalg.norm(g - gx) <= TOL * np.linalg.norm(gx) + sl, (n, gx.shape)
        off += gx.size
    assert off == grad.size
