"""GPU: projections at the ends of the number range: weights whose sum overflows, atoms that are points,
weights that are not finite."""
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


def _ball(rng, n, radius):
    g = rng.standard_normal((n, 3))
    g *= (radius * rng.random(n) ** (1 / 3) / np.linalg.norm(g, axis=1))[:, None]
    return np.concatenate([g, np.ones((n, 1))], 1).astype(np.float32)


@pytest.mark.parametrize("npix", [32, 96, 128, 192])
def test_weights_whose_sum_overflows(env, npix):
    """Weights of 2^116: their sum, the DC coefficient alone, exceeds the FP32 range, so ln L changes by ln of the
    scale.  1e-3, the FP32 form's bound: the spectra's norms are near 2^127, and the FP32 factor that takes
    them to 1 has lost bits to underflow."""
    bioem, ctx = env
    rng = np.random.default_rng(npix)
    pixel, n, bits = 128.0 / npix, 5000, 116
    assert n * 2.0 ** bits > float(np.finfo(np.float32).max)
    atoms = _ball(rng, n, 40.0)
    quats = rng.standard_normal((3, 4)).astype(np.float32)
    ctfs = [(1.0e4, 0.1, 0.0, 300.0), (2.0e4, 0.2, 30.0, 300.0)]
    im = bioem.prepare_images(ctx, _dev(rng.standard_normal((2, npix, npix)).astype(np.float32)), pixel)
    out = []
    for scale in (1.0, 2.0 ** bits):
        a = atoms.copy()
        a[:, 3] *= np.float32(scale)
        ps = bioem.project_model(ctx, _dev(a), 1.5, _dev(quats), ctfs, npix, pixel)
        out.append([x.cpu().numpy() for x in bioem.score_pairs(ctx, im, ps, 3)])
        assert ctx.status() == 0
    for one, two in zip(*out):
        assert np.isfinite(one).all()
        np.testing.assert_allclose(two, one - bits * np.log(2.0), rtol=0, atol=1e-3)


IDENTITY = np.array([[1, 0, 0, 0]], dtype=np.float32)


@pytest.mark.parametrize("npix", [32, 64, 96, 128, 192])
@pytest.mark.parametrize("sigma_px", [1e-3, 1e-4, 1e-6, 1e-7, 1e-8])
def test_atoms_that_are_points(env, npix, sigma_px):
    """Atoms on pixel boundaries and up to 2^-8 pixels beside them, narrower than the FP32 spacing of their
    positions in units of sigma.  The bound of the maps of any window: 2e-5 of the largest value."""
    bioem, ctx = env
    rng = np.random.default_rng(npix)
    atoms = np.zeros((300, 4), dtype=np.float32)
    atoms[:, :2] = rng.integers(2, npix - 2, (300, 2)) - npix / 2 - 0.5
    atoms[150:, :2] += rng.choice([-1, 1], (150, 2)) * 2.0 ** -rng.integers(8, 18, (150, 1))
    atoms[:, 3] = rng.uniform(0.5, 1.5, 300)
    ctf = (0.0, 1.0, 0.0, 300.0)
    got = bioem.synthetic_maps(ctx, _dev(atoms), sigma_px, _dev(IDENTITY), [ctf], npix, 1.0).cpu().numpy()[0]
    want = oracle.apply_psf(oracle.project(atoms, IDENTITY[0], sigma_px, npix, 1.0), ctf, 1.0)
    assert ctx.status() == 0
    np.testing.assert_allclose(got, want, rtol=0, atol=2e-5 * np.abs(want).max())


@pytest.mark.parametrize("npix", [32, 96, 128, 192])
@pytest.mark.parametrize("weight", [np.nan, np.inf, -np.inf])
def test_weights_that_are_not_finite(env, npix, weight):
    """An atom whose weight is not finite makes the projection degenerate (NUMERIC) and the map undefined
    wherever it lies beside the image's columns: its weight meets the zeros there.  Far above or below the
    image, where no row comes near it, it has no part in either."""
    bioem, ctx = env
    rng = np.random.default_rng(npix)
    for x, y, part in ((0, 0, True), (5 * npix, 0, True), (0.5 * npix + 16.2, 3, True), (2, 0.5 * npix + 11.2, True),
                       (0, 5 * npix, False), (-5 * npix, 5 * npix, False)):
        atoms = rng.uniform(-8, 8, (40, 4)).astype(np.float32)
        atoms[:, 3] = 1.0
        atoms[7] = (x, y, 0.0, weight)
        bioem.project_model(ctx, _dev(atoms), 1.0, _dev(IDENTITY), [(1.0e4, 0.1, 0.0, 300.0)], npix, 1.0)
        assert ctx.status() == (bioem.ERR_NUMERIC if part else 0), (x, y)
        got = bioem.synthetic_maps(ctx, _dev(atoms), 1.0, _dev(IDENTITY), [(1.0e4, 0.1, 0.0, 300.0)], npix, 1.0).cpu().numpy()
        assert np.isfinite(got).any() != part and np.isfinite(got).all() != part, (x, y)


@pytest.mark.parametrize("npix", [32, 64, 96, 128, 192])
@pytest.mark.parametrize("top", [1e37, 2e38, 3e38])
def test_maps_up_to_the_largest_numbers(env, npix, top):
    """N^2 times the largest value of the map (what the unscaled inverse transform reaches) up to 3e38.  The
    bound of the maps of any window: 2e-5 of the largest value."""
    bioem, ctx = env
    atoms = np.array([[1.3, -2.1, 0.0, 1.0]], dtype=np.float32)
    want = -oracle.project(atoms, IDENTITY[0], 1.5, npix, 1.0)   # defocus 0, amplitude contrast 1: CTF = -1
    atoms[0, 3] = top / (npix * npix * np.abs(want).max())
    got = bioem.synthetic_maps(ctx, _dev(atoms), 1.5, _dev(IDENTITY), [(0.0, 1.0, 0.0, 300.0)], npix, 1.0).cpu().numpy()[0]
    want *= float(atoms[0, 3])
    np.testing.assert_allclose(got.astype(np.float64), want, rtol=0, atol=2e-5 * np.abs(want).max())
