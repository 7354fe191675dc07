"""GPU: per-pair values of an image that is not finite."""
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


@pytest.mark.parametrize("npix,shift", [(32, 4), (64, 4), (64, 8), (96, 12), (128, 4)])
def test_pairs_of_an_undefined_image(env, npix, shift):
    """A NaN pixel: NUMERIC, and ln L = -inf for each of the image's pairs, in score_pairs and in its own list;
    the other images' values are those of a stack without it."""
    import torch
    bioem, ctx = env
    cfg = workloads.get_config("tiny", npix=npix, pixel_A=64.0 / npix, max_shift=shift, n_orient=23, n_defocus=1,
                               bfactors=(0.0,), n_atoms=60)
    wl = workloads.workload(cfg, n_img=1)
    imgs = np.random.default_rng(npix).standard_normal((3, npix, npix)).astype(np.float32)
    imgs[1, 2, 3] = np.nan
    im = bioem.prepare_images(ctx, _dev(imgs), cfg.pixel_A)
    good = bioem.prepare_images(ctx, _dev(imgs[[0, 2]]), cfg.pixel_A)
    assert ctx.status() == bioem.ERR_NUMERIC
    ps = bioem.project_model(ctx, _dev(wl["atoms"]), cfg.sigma_A, _dev(wl["quats"]), wl["ctfs"], npix, cfg.pixel_A)
    off, idx = _dev(np.array([0, 7, 30, 40], dtype=np.int32)), _dev((np.arange(40) % 23).astype(np.int32))
    for s in (shift, shift // 2):
        pmax, plse = bioem.score_pairs(ctx, im, ps, s)
        gmax, glse = bioem.score_pairs(ctx, good, ps, s)
        listed = bioem.score_gathered_pairs(ctx, im, ps, s, off, idx, 23)
        for v in (pmax[1], plse[1], listed[7:30]):
            assert bool((v == float("-inf")).all())
        assert torch.equal(pmax[[0, 2]], gmax) and torch.equal(plse[[0, 2]], glse)
        assert bool(torch.isfinite(listed[:7]).all()) and bool(torch.isfinite(listed[30:]).all())
    assert ctx.status() == 0
