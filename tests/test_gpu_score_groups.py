"""GPU: the FP32 scoring instances at the edges of their group batches, and the reductions over parts and
waves, each against the float64 oracle or against a run that is cut differently."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
TOL = 1e-3   # ln P and ln L of the FP32 form against float64 (the other parity tests' bound)


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


def _case(npix, shift, n_img, n_orient, n_defocus=1, bfactors=(0.0,)):
    cfg = workloads.get_config("tiny", npix=npix, pixel_A=64.0 / npix, max_shift=shift, n_orient=n_orient,
                               n_defocus=n_defocus, bfactors=bfactors, n_atoms=60)
    wl = workloads.workload(cfg, n_img=n_img)
    return cfg, wl, oracle.synthesize_images(wl)


# every instance (image size, window of the instance) and, at 128 px, both
@pytest.mark.parametrize("npix,shift", [(32, 4), (64, 4), (64, 8), (96, 12), (128, 4), (128, 16), (192, 24)])
def test_pairs_at_batch_edges(env, npix, shift):
    """Per-pair values of 1 .. 43 sets (below, at and above a group's and a block's batch) are those of the
    whole range bit for bit, for the full window and a smaller one, and agree with the oracle."""
    bioem, ctx = env
    n = 97
    cfg, wl, imgs = _case(npix, shift, 2, n)
    im = bioem.prepare_images(ctx, _dev(imgs), cfg.pixel_A)
    ps = bioem.project_model(ctx, _dev(wl["atoms"]), cfg.sigma_A, _dev(wl["quats"]), wl["ctfs"], npix, cfg.pixel_A)
    few = 6
    for s in (shift, shift // 2):
        pmax, plse = bioem.score_pairs(ctx, im, ps, s)
        for begin, count in ((0, 1), (3, 2), (5, 7), (1, 8), (0, 11), (40, 16), (0, 25), (10, 33), (54, 43)):
            a, b = bioem.score_pairs(ctx, im, ps, s, begin, count)
            assert (a == pmax[:, begin:begin + count]).all() and (b == plse[:, begin:begin + count]).all(), (begin, count)
        if npix <= 128:
            ref = oracle.score(imgs, wl["atoms"], wl["quats"][:few], wl["ctfs"], cfg.sigma_A, cfg.pixel_A, s)
            np.testing.assert_allclose(pmax.cpu().numpy()[:, :few], ref["pair_max"], rtol=0, atol=TOL)
            np.testing.assert_allclose(plse.cpu().numpy()[:, :few], ref["pair_lse"], rtol=0, atol=TOL)
    assert ctx.status() == 0


# 1 image is cut into the most parts, 40 images x 2 defocus into few; 3 PSFs make no multiple of the
# reduction's groups of four
@pytest.mark.parametrize("n_img,n_defocus,bfactors", [(1, 3, (0.0,)), (3, 1, (0.0,)), (40, 2, (0.0, 50.0))])
def test_reduction_parts_and_waves(env, n_img, n_defocus, bfactors):
    """ln P, per-orientation ln P and the maximising parameters from one wave in parts, from many waves, and
    from the allocation-free call, against the oracle and against one another.  The float64 sums differ in
    order only: 1e-9 covers that for values below 1e5."""
    import torch
    bioem, ctx = env
    cfg, wl, imgs = _case(32, 4, n_img, 600, n_defocus, bfactors)
    im = bioem.prepare_images(ctx, _dev(imgs), cfg.pixel_A)
    ps = bioem.project_model(ctx, _dev(wl["atoms"]), cfg.sigma_A, _dev(wl["quats"]), wl["ctfs"], 32, cfg.pixel_A)
    one = bioem.score_all(ctx, im, ps, 4, per_orient=True, best=True)
    out = torch.empty(n_img, dtype=torch.float64, device="cuda:0")
    bioem.score_noalloc(ctx, im, ps, 4, out)
    try:
        ctx.set_scratch_limit(max(4096, n_img * 12 * 70))   # about 70 sets per wave
        many = bioem.score_all(ctx, im, ps, 4, per_orient=True, best=True)
    finally:
        ctx.set_scratch_limit(2 << 30)
    assert ctx.status() == 0
    for k in ("logP", "logP_orient"):
        np.testing.assert_allclose(many[k].cpu().numpy(), one[k].cpu().numpy(), rtol=0, atol=1e-9)
    for k in ("best_q", "best_ctf", "best_dx", "best_dy", "best_logL"):
        assert (many[k] == one[k]).all(), k
    np.testing.assert_allclose(out.cpu().numpy(), one["logP"].cpu().numpy(), rtol=0, atol=1e-9)
    ref = oracle.score(imgs[:3], wl["atoms"], wl["quats"], wl["ctfs"], cfg.sigma_A, cfg.pixel_A, 4)
    np.testing.assert_allclose(one["logP"].cpu().numpy()[:3], ref["logP"], rtol=0, atol=TOL)
    np.testing.assert_allclose(one["logP_orient"].cpu().numpy()[:3], ref["logP_orient"], rtol=0, atol=TOL)
    np.testing.assert_allclose(one["best_logL"].cpu().numpy()[:3], [b[4] for b in ref["best"]], rtol=0, atol=TOL)


# more spectra than one phase (or several chunks, at the +-16 px window), images fewer than, near and above the
# number of SMs, so that blocks get parts of one image, two images, or several
@pytest.mark.parametrize("npix,shift,n_img,n_orient", [
    (32, 4, 37, 1500), (64, 4, 41, 420), (64, 8, 153, 420), (96, 12, 29, 331), (128, 4, 37, 201), (128, 4, 1, 201),
    (128, 4, 307, 13), (128, 16, 37, 201)])
def test_whole_range_equals_its_parts(env, npix, shift, n_img, n_orient):
    """Per-pair values of a long range are, bit for bit, those of short ranges of the same sets."""
    bioem, ctx = env
    cfg, wl, _ = _case(npix, shift, 1, n_orient, 4, (0.0, 50.0))
    imgs = np.random.default_rng(npix + n_img).standard_normal((n_img, npix, npix)).astype(np.float32)
    im = bioem.prepare_images(ctx, _dev(imgs), cfg.pixel_A)
    ps = bioem.project_model(ctx, _dev(wl["atoms"]), cfg.sigma_A, _dev(wl["quats"]), wl["ctfs"], npix, cfg.pixel_A)
    n_ps = n_orient * 8
    pmax, plse = bioem.score_pairs(ctx, im, ps, shift)
    for begin in range(0, n_ps, 333):
        count = min(333, n_ps - begin)
        a, b = bioem.score_pairs(ctx, im, ps, shift, begin, count)
        assert (a == pmax[:, begin:begin + count]).all() and (b == plse[:, begin:begin + count]).all(), begin
    assert bool((pmax == pmax).all()) and ctx.status() == 0


# empty lists first, last and between; one image alone; lists far longer than the others; fewer sets than blocks
@pytest.mark.parametrize("npix,shift,lengths", [
    (32, 4, [0, 0, 700, 1, 0, 3, 0]), (64, 8, [2100]), (96, 12, [1, 0, 1]), (128, 4, [5, 900, 0, 40, 1, 1, 260] * 9),
    (128, 16, [0, 33, 2, 1000, 0, 7] * 30)])
def test_gathered_lists_of_any_length(env, npix, shift, lengths):
    """Each image against its own list: the values of the whole range's pairs, bit for bit."""
    import torch
    bioem, ctx = env
    cfg, wl, _ = _case(npix, shift, 1, 150)
    n_img = len(lengths)
    rng = np.random.default_rng(npix)
    im = bioem.prepare_images(ctx, _dev(rng.standard_normal((n_img, npix, npix)).astype(np.float32)), cfg.pixel_A)
    ps = bioem.project_model(ctx, _dev(wl["atoms"]), cfg.sigma_A, _dev(wl["quats"]), wl["ctfs"], npix, cfg.pixel_A)
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    idx = rng.integers(0, 150, off[-1]).astype(np.int32)
    got = bioem.score_gathered_pairs(ctx, im, ps, shift, _dev(off), _dev(idx), max(lengths))
    _, plse = bioem.score_pairs(ctx, im, ps, shift)
    rows = torch.from_numpy(np.repeat(np.arange(n_img), lengths)).to(plse.device)
    want = plse[rows, _dev(idx).long()]
    # the pair sums of the two calls round ln L in a different order: float64, values below 1e5
    assert float((got - want).abs().max()) < 1e-9 and ctx.status() == 0
