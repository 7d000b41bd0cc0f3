"""The denoiser's fused element-wise kernels (pooling, up-sampling into the decoder's inputs, masked gradients with
their bias sums, the optimiser over all layers) on images that are not square and batches that are not powers of two:
whole-network gradients of a network whose values all fit BF16, and one optimiser step in closed form."""

import numpy as np
import pytest

from oracle import nn

pytestmark = pytest.mark.gpu


def _pair(rng, n, h, w):
    yy, xx = np.mgrid[0:h, 0:w] / h
    clean = np.stack([1.0 + 0.5 * np.sin(3 * a * xx + b) * np.cos(3 * c * yy + d) for a, b, c, d in rng.uniform(0.5, 2, (n, 4))])
    return clean, clean * rng.gamma(20.0, 1 / 20.0, size=clean.shape)


def _exact_net(rng):
    """One non-zero weight per output channel, a power of two: activations keep their inputs' few mantissa bits and
    every forward and input-gradient sum is exact in FP32, so BF16 roundings cannot differ from the oracle's."""
    out = []
    for i, (ci, co) in enumerate(zip(nn.CIN, nn.COUT)):
        w = np.zeros((co, 9, ci))
        src = rng.integers(0, 1 if i == 0 else ci, co)
        w[np.arange(co), rng.integers(0, 9, co), src] = rng.choice([1.0, 1.0, 0.5, 2.0, -1.0], co)
        out.append((w, rng.choice([0.0, 0.0, 0.5], co)))
    return out


@pytest.mark.parametrize("h,w,n", [(16, 16, 1), (16, 48, 2), (64, 96, 1), (112, 64, 3)])
def test_exact_network(gpu, h, w, n):
    """Gradients of all layers within the FP32 rounding of their sums over n h w pixels (and many equal values in the
    pooling windows: the first one takes the gradient)."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(h + w)
    weights = _exact_net(rng)
    c = gpu.Context(0)
    c.denoise_init(h, w, n, seed=1)
    for i, (wt, b) in enumerate(weights):
        c.denoise_set_layer(i, wt, b)
    # half the pixels 0.5, half 1.5: the mean is 1, so the normalised image is the image
    noisy = np.stack([rng.permutation(np.repeat([0.5, 1.5], h * w // 2)).reshape(h, w) for _ in range(n)])
    clean = rng.choice([0.5, 1.0, 2.0], noisy.shape)
    loss = c.denoise_train_step(torch.tensor(noisy, dtype=torch.float32).cuda(),
                                torch.tensor(clean, dtype=torch.float32).cuda(), lr=0.0)
    ref_loss, grads = nn.UNet(weights, bf16=True).loss_and_grads(noisy, clean)
    assert abs(loss / ref_loss - 1.0) < 1e-6
    for i in range(15):
        _, _, gw, gb = c.denoise_layer(i)
        for got, ref in ((gw, grads[i][0]), (gb, grads[i][1])):
            assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max(), i


def test_optimiser_step(gpu):
    """The first Adam step moves every parameter by lr g / (|g| + 1e-8) (its moments are g and g^2 after bias
    correction, to a few FP32 roundings), and the operand copies hold the new weights: a network set to them gives the
    same images."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(3)
    c = gpu.Context(0)
    c.denoise_init(32, 48, 2, seed=4)
    before = [c.denoise_layer(i)[:2] for i in range(15)]
    clean, noisy = (torch.tensor(t, dtype=torch.float32).cuda() for t in _pair(rng, 2, 32, 48))
    lr = 1e-3
    c.denoise_train_step(noisy, clean, lr)
    d = gpu.Context(0)
    d.denoise_init(32, 48, 2, seed=9)
    for i in range(15):
        w, b, gw, gb = c.denoise_layer(i)
        for p0, p1, g in ((before[i][0], w, gw), (before[i][1], b, gb)):
            g = g.astype(np.float64)
            step = lr * g / (np.abs(g) + 1e-8)
            # 1e-8 is added to sqrt(v / c2), which carries a few roundings of |g|
            assert np.abs((p0 - p1) - step).max() <= 1e-5 * lr + 2.0**-23 * np.abs(p0).max()
        d.denoise_set_layer(i, w, b)
    assert torch.equal(c.denoise_infer(noisy), d.denoise_infer(noisy))
