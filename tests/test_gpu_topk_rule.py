"""GPU: short proposals (one pass over the scores per pick) against longer ones (selection and sort)."""
import pytest

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


# both sides of the rule's lines: 3 and 4 picks, 8 and 9, 2,048 and 2,049 bins
@pytest.mark.parametrize("nq,nd,short,long", [(512, 4, 8, 9), (683, 3, 3, 4), (683, 3, 8, 30), (40, 1, 8, 40), (3000, 2, 3, 64), (5, 1, 1, 5)])
@pytest.mark.parametrize("ties", [False, True])
def test_short_proposals_begin_the_long_ones(env, nq, nd, short, long, ties):
    import torch
    bioem, ctx = env
    net = bioem.CNN(ctx, image_px=16, downsample=2, channels=4, n_qbins=nq, n_dbins=nd, max_batch=4, seed=3)
    gen = torch.Generator(device="cuda:0").manual_seed(nq)
    theta = torch.randn(net.n_params, generator=gen, device="cuda:0") * 0.3
    if ties:   # scores on few values
        theta = (theta * 2).round() / 2
    net.set_params(theta)
    imgs = torch.randn((6, 16, 16), generator=gen, device="cuda:0")
    b1, s1 = net.propose(imgs, short)
    b2, s2 = net.propose(imgs, long)
    assert torch.equal(b1, b2[:, :short]) and torch.equal(s1, s2[:, :short])
