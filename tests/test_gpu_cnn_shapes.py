"""GPU: the proposal network's kernels where their tiles end: image sizes and channel counts that are no
multiple of a thread's or a block's share, column tiles beyond the first, and the top-k at the edges of
its sorting network, with equal and undefined scores."""
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


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")


# (image px, downsample, channels, orientation bins, defocus bins, batch): 8 px leaves 1 px outputs; 24 px
# rows are no whole groups of four at the last layers; 33 and 64 channels take a second channel block;
# 72 px rows take a second column tile of the weight gradients
@pytest.mark.parametrize("px,down,C,nq,nd,B", [(8, 1, 3, 5, 1, 2), (24, 1, 5, 70, 3, 3), (32, 1, 33, 9, 2, 2),
                                               (32, 1, 64, 130, 64, 1), (144, 2, 4, 7, 5, 2), (64, 1, 17, 65, 4, 67)])
def test_network_shapes(env, px, down, C, nq, nd, B):
    """Logits, losses and gradients against float64.  Tolerance: the sums run over at most a few 1e5
    FP32 terms (relative error below 1e-4); a ReLU input that rounds across zero moves a gradient by a
    share of one sample's part, below the 2e-3 that the other network tests allow."""
    bioem, ctx = env
    rng = np.random.default_rng(100 + px + C)
    net = bioem.CNN(ctx, image_px=px, downsample=down, channels=C, n_qbins=nq, n_dbins=nd, max_batch=B, seed=1)
    _, _, _, n = ocnn.layout(px // down, C, nq, nd)
    theta = (rng.standard_normal(n) * (1.5 / np.sqrt(9 * C))).astype(np.float16).astype(np.float64)
    imgs = rng.standard_normal((B, px, px)).astype(np.float32)
    yq, yd = rng.integers(0, nq, B).astype(np.int32), rng.integers(0, nd, B).astype(np.int32)
    net.set_params(_dev(theta.astype(np.float32)))
    lq, ld = net.forward(_dev(imgs))
    g, loss = net.gradients(_dev(imgs), _dev(yq), _dev(yd))
    want_loss, want_g = ocnn.loss_and_grad(theta, imgs.astype(np.float64), yq, yd, down, C, nq, nd)
    wq, wd, _ = ocnn.forward(theta, imgs.astype(np.float64), down, C, nq, nd)
    np.testing.assert_allclose(lq.cpu().numpy(), wq, rtol=0, atol=1e-4 * np.abs(wq).max())
    np.testing.assert_allclose(ld.cpu().numpy(), wd, rtol=0, atol=1e-4 * np.abs(wd).max())
    np.testing.assert_allclose(loss.cpu().numpy(), want_loss, rtol=2e-4)
    offs, heads, _, _ = ocnn.layout(px // down, C, nq, nd)
    got = g.cpu().numpy().astype(np.float64)
    for off, shape in [o for pair in offs for o in pair] + list(heads):
        sl = slice(off, off + int(np.prod(shape)))
        err = np.linalg.norm(got[sl] - want_g[sl]) / max(np.linalg.norm(want_g[sl]), 1e-12)
        assert err < 2e-3, (off, shape, err)


# sorting networks of 64 (the smallest), 128, 2048 and 4096 entries, whole and partly filled; 70,000 bins
# do not fit the sorted form (16-bit bins)
@pytest.mark.parametrize("nq,nd,k", [(40, 4, 1), (40, 4, 63), (40, 4, 64), (40, 4, 65), (40, 4, 160), (700, 3, 2049),
                                     (700, 3, 2100), (1300, 4, 4096), (35000, 2, 5)])
def test_propose_order(env, nq, nd, k):
    """The k best joint bins: distinct, best first, equal scores by bin, none better left out.  Scores are
    FP32 sums of two log-softmaxes below 32 in size: 1e-5 covers their rounding."""
    bioem, ctx = env
    rng = np.random.default_rng(nq + k)
    net = bioem.CNN(ctx, image_px=16, downsample=2, channels=4, n_qbins=nq, n_dbins=nd, max_batch=3, seed=2)
    theta = (rng.standard_normal(net.n_params) * 0.4).astype(np.float16)
    net.set_params(_dev(theta.astype(np.float32)))
    imgs = _dev(rng.standard_normal((4, 16, 16)).astype(np.float32))
    bins, scores = net.propose(imgs, k)
    logits = [net.forward(imgs[i:i + 3]) for i in (0, 3)]
    lq = np.concatenate([x[0].cpu().numpy() for x in logits]).astype(np.float64)
    ld = np.concatenate([x[1].cpu().numpy() for x in logits]).astype(np.float64)
    joint = (ocnn.log_softmax(lq)[:, :, None] + ocnn.log_softmax(ld)[:, None, :]).reshape(4, -1)
    bins, scores = bins.cpu().numpy(), scores.cpu().numpy()
    for i in range(4):
        assert len(set(bins[i])) == k and bins[i].min() >= 0 and bins[i].max() < nq * nd
        np.testing.assert_allclose(scores[i], joint[i][bins[i]], rtol=0, atol=1e-5)
        step = np.diff(scores[i])
        assert np.all(step <= 0) and np.all(np.diff(bins[i])[step == 0] > 0)
        rest = np.delete(joint[i], bins[i])
        assert rest.size == 0 or rest.max() <= scores[i, -1] + 1e-5


def test_propose_equal_and_undefined_scores(env):
    """Zero weights: every score is equal, so the lowest bins in order.  A NaN bias of the last
    orientation bin makes every log-softmax undefined: no bin (0x7fffffff at -inf)."""
    import torch
    bioem, ctx = env
    nq, nd = 300, 4
    net = bioem.CNN(ctx, image_px=16, downsample=2, channels=4, n_qbins=nq, n_dbins=nd, max_batch=3, seed=2)
    theta = torch.zeros(net.n_params, device="cuda:0")
    net.set_params(theta)
    imgs = torch.randn((3, 16, 16), device="cuda:0")
    for k in (1, 70, 1199, 1200):
        bins, scores = net.propose(imgs, k)
        assert torch.equal(bins.cpu(), torch.arange(k, dtype=torch.int32).expand(3, k))
        assert torch.unique(scores).numel() == 1
    _, heads, _, _ = ocnn.layout(8, 4, nq, nd)
    theta[heads[1][0] + nq - 1] = float("nan")
    net.set_params(theta)
    bins, scores = net.propose(imgs, 90)
    assert bool((bins == 0x7FFFFFFF).all()) and bool((scores == float("-inf")).all())
