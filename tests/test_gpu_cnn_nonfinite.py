"""GPU: images whose inputs to the network are not finite stay out of the other images' gradients."""
import numpy as np
import pytest

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_06634_gb300 as bioem
    from paper_1609_06634_gb300 import build
    build.build()
    return bioem, bioem.Context(0)


def _gradients(net, theta, imgs, yq, yd):
    import torch
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")
    net.set_params(dev(theta))
    g, loss = net.gradients(dev(imgs), dev(yq), dev(yd))
    return g.cpu().numpy(), loss.cpu().numpy()


# rows of whole groups of four and not (the last layers of 40 px), one and two column tiles and channel blocks
@pytest.mark.parametrize("px,down,C", [(64, 1, 8), (40, 1, 35), (144, 1, 4)])
@pytest.mark.parametrize("bad", ["nan", "inf", "overflow"])
def test_images_that_are_not_finite(env, px, down, C, bad):
    """With zero biases, an image with a NaN or infinite pixel gives first activations of 0, as an image without
    contrast does: the batch's gradients and losses are the same bit for bit.  So is an image too faint to
    standardise (inputs of +-inf) where the weights of some layer are all negative: its activations are +inf
    before that layer and 0 from it on, and every gradient that meets them is 0."""
    bioem, ctx = env
    B, nq, nd = 5, 9, 3
    offs, heads, _, n = ocnn.layout(px // down, C, nq, nd)
    rng = np.random.default_rng(px + C)
    theta = (rng.standard_normal(n) * (1.5 / np.sqrt(9 * C))).astype(np.float16).astype(np.float32)
    for (_, _), (off, shape) in offs:
        theta[off:off + int(np.prod(shape))] = 0.0
    imgs = rng.standard_normal((B, px, px)).astype(np.float32)
    yq, yd = rng.integers(0, nq, B).astype(np.int32), rng.integers(0, nd, B).astype(np.int32)
    net = bioem.CNN(ctx, image_px=px, downsample=down, channels=C, n_qbins=nq, n_dbins=nd, max_batch=B, seed=1)
    plain = imgs.copy()
    plain[2] = 0.0
    thetas = [theta]
    if bad == "overflow":
        faint = np.where(np.arange(px) < px // 2, 1e-43, -1e-43).astype(np.float32)
        imgs[2] = faint[None, :]
        thetas = []
        for layer in range(1, 6):   # positive weights up to it, negative ones there
            t = theta.copy()
            for k in range(layer + 1):
                off, shape = offs[k][0]
                w = t[off:off + int(np.prod(shape))]
                w[:] = np.maximum(np.abs(w), 1e-3) * (1.0 if k < layer else -1.0)
            thetas.append(t)
    else:
        imgs[2, 3, 5] = np.float32(bad)
    for t in thetas:
        g, loss = _gradients(net, t, imgs, yq, yd)
        want_g, want_loss = _gradients(net, t, plain, yq, yd)
        assert np.isfinite(want_g).all() and np.isfinite(want_loss).all()
        np.testing.assert_array_equal(loss, want_loss)
        np.testing.assert_array_equal(g, want_g)
