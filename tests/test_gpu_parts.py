"""GPU: many images of few parameter sets, where the blocks' parts end on whole rounds of a block."""
import numpy as np
import pytest

import workloads

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


# one round per image (1 .. a block's pairs), one set more, and three rounds; images below, at and above the
# number of SMs
@pytest.mark.parametrize("npix,shift,pairs", [(32, 4, 90), (64, 8, 27), (96, 12, 15), (128, 4, 20)])
@pytest.mark.parametrize("n_img", [100, 152, 307])
def test_many_images_of_few_sets(env, npix, shift, pairs, n_img):
    """Per-pair values of all images at once, and of lists of those lengths, are bit for bit those of ten images at
    a time (which are cut into single batches)."""
    import torch
    bioem, ctx = env
    cfg = workloads.get_config("tiny", npix=npix, pixel_A=64.0 / npix, max_shift=shift, n_orient=3 * pairs, n_defocus=1,
                               bfactors=(0.0,), n_atoms=60)
    wl = workloads.workload(cfg, n_img=1)
    rng = np.random.default_rng(npix + n_img)
    imgs = _dev(rng.standard_normal((n_img, npix, npix)).astype(np.float32))
    im = bioem.prepare_images(ctx, imgs, cfg.pixel_A)
    ps = bioem.project_model(ctx, _dev(wl["atoms"]), cfg.sigma_A, _dev(wl["quats"]), wl["ctfs"], npix, cfg.pixel_A)
    n_ps = 3 * pairs
    full = torch.cat([bioem.score_pairs(ctx, bioem.prepare_images(ctx, imgs[i:i + 10], cfg.pixel_A), ps, shift)[1]
                      for i in range(0, n_img, 10)])
    for count in (1, pairs // 2 + 1, pairs, pairs + 1, n_ps):
        pmax, plse = bioem.score_pairs(ctx, im, ps, shift, 0, count)
        assert torch.equal(plse, full[:, :count]), count
        off = np.arange(n_img + 1) * count
        off[1:] -= (np.arange(1, n_img + 1) % 3 == 0) * (count // 2)   # two lengths, whole and uneven
        off = np.maximum.accumulate(off).astype(np.int32)
        lens = np.diff(off)
        idx = np.concatenate([np.arange(k) % n_ps for k in lens]).astype(np.int32)
        got = bioem.score_gathered_pairs(ctx, im, ps, shift, _dev(off), _dev(idx), int(lens.max()))
        rows = _dev(np.repeat(np.arange(n_img), lens))
        # the pair sums of the two calls round ln L in a different order: float64, values below 1e5
        assert float((got - full[rows, _dev(idx).long()]).abs().max()) < 1e-9, count
    assert ctx.status() == 0
