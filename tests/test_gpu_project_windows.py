"""GPU: projection and transforms where their windows and tiles end, against the float64 oracle."""
import numpy as np
import pytest

import oracle

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


# atoms: none of a second chunk (31), exactly one chunk, one more, several; sigma of 0.05 to 30 pixels: windows
# of a few pixels up to the whole image
@pytest.mark.parametrize("npix", [32, 64, 96, 128, 192])
@pytest.mark.parametrize("n_atoms,sigma_px", [(1, 0.7), (31, 0.05), (32, 1.4), (33, 4.0), (200, 30.0)])
def test_maps_of_any_window(env, npix, n_atoms, sigma_px):
    """Maps of atoms inside, across and far outside the box, with positive and negative weights.  FP32 sums
    of at most 200 products and transforms of N^2 <= 36,864 terms: 2e-5 of the largest value."""
    bioem, ctx = env
    rng = np.random.default_rng(npix + n_atoms)
    pixel = 1.3
    box = npix * pixel
    atoms = np.empty((n_atoms, 4), dtype=np.float32)
    atoms[:, :3] = rng.uniform(-0.6 * box, 0.6 * box, (n_atoms, 3))
    atoms[:, 3] = rng.uniform(-1.0, 2.0, n_atoms)
    if n_atoms > 2:
        atoms[1, :3] = (50.0 * box, 0.0, 0.0)          # its window lies off the image
        atoms[2, :3] = 0.0
    quats = rng.standard_normal((3, 4)).astype(np.float32)
    ctfs = [(1.0e4, 0.1, 0.0, 300.0), (2.0e4, 0.3, 40.0, 200.0), (0.0, 1.0, 10.0, 300.0)]
    got = bioem.synthetic_maps(ctx, _dev(atoms), sigma_px * pixel, _dev(quats), ctfs, npix, pixel).cpu().numpy()
    assert ctx.status() == 0
    for i in range(3):
        want = oracle.apply_psf(oracle.project(atoms, quats[i], sigma_px * pixel, npix, pixel), ctfs[i], pixel)
        np.testing.assert_allclose(got[i], want, rtol=0, atol=2e-5 * max(np.abs(want).max(), 1e-3))


def test_images_that_are_not_16_byte_aligned(env):
    """A view that starts on a 4-byte boundary gives the handle that its aligned copy gives."""
    import torch
    bioem, ctx = env
    flat = torch.randn(3 * 32 * 32 + 1, device="cuda:0")
    quats, atoms = _dev(np.eye(4, dtype=np.float32)), torch.randn((40, 4), device="cuda:0") * 8.0
    atoms[:, 3] = 1.0
    ps = bioem.project_model(ctx, atoms, 1.5, quats, [(1.0e4, 0.1, 0.0, 300.0)], 32, 2.0)
    view = flat[1:].view(3, 32, 32)
    assert view.data_ptr() % 16 == 4
    a = bioem.score(ctx, bioem.prepare_images(ctx, view, 2.0), ps, 4)
    b = bioem.score(ctx, bioem.prepare_images(ctx, view.clone(), 2.0), ps, 4)
    assert ctx.status() == 0 and torch.equal(a, b)


# 17 PSFs: one more than are reduced together
@pytest.mark.parametrize("npix,n_defocus", [(32, 17), (96, 1), (192, 2)])
def test_scores_of_many_psfs(env, npix, n_defocus):
    """Unit-norm spectra and ln B of every PSF through per-pair ln L against the oracle (1e-3: the FP32 form)."""
    bioem, ctx = env
    rng = np.random.default_rng(npix)
    pixel = 64.0 / npix
    atoms = np.concatenate([rng.uniform(-15, 15, (80, 3)), np.ones((80, 1))], 1).astype(np.float32)
    quats = rng.standard_normal((3, 4)).astype(np.float32)
    ctfs = np.array([(d, 0.1, 20.0, 300.0) for d in np.linspace(0.5e4, 2.5e4, n_defocus)])
    base = oracle.apply_psf(oracle.project(atoms, quats[1], 1.5, npix, pixel), ctfs[0], pixel)
    imgs = (base[None] / base.std() + 2.0 * rng.standard_normal((2, npix, npix))).astype(np.float32)
    im = bioem.prepare_images(ctx, _dev(imgs), pixel)
    ps = bioem.project_model(ctx, _dev(atoms), 1.5, _dev(quats), ctfs, npix, pixel)
    pmax, plse = bioem.score_pairs(ctx, im, ps, 2)
    assert ctx.status() == 0
    ref = oracle.score(imgs, atoms, quats, ctfs, 1.5, pixel, 2)
    np.testing.assert_allclose(pmax.cpu().numpy(), ref["pair_max"], rtol=0, atol=1e-3)
    np.testing.assert_allclose(plse.cpu().numpy(), ref["pair_lse"], rtol=0, atol=1e-3)
