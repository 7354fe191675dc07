"""GPU: the batched launch where its chunks and pair batches end, 192 px above all (an instance of its own,
two pairs in flight), and lists at 192 px."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
TOL = 1e-3   # ln P of the FP32 form against float64 (the other parity tests' bound)


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


def _case(npix, n_sets, n_img):
    cfg = workloads.get_config("tiny", npix=npix, pixel_A=64.0 / npix, max_shift=npix // 8, n_orient=n_sets, n_defocus=1,
                               bfactors=(0.0,), n_atoms=60)
    wl = workloads.workload(cfg, n_img=n_img)
    return cfg, wl, oracle.synthesize_images(wl)


# sets: one, fewer and more than a pair batch, one more than the default chunk of a few images at 192 px (16)
@pytest.mark.parametrize("n_sets", [1, 3, 17])
@pytest.mark.parametrize("share", [0.0, 0.5, 1.0])
def test_ragged_batches(env, n_sets, share):
    """Two models against stacks of 192 and of 64, 96 and 128 px with odd numbers of sets, windows of 0, half and
    the whole of each size's instance, against the oracle (1e-3 and the float32 output's rounding)."""
    bioem, ctx = env
    stacks, projsets, refs, shifts = [], [[], []], [[], []], []
    for npix in (192, 64, 96, 128):
        shift = int(share * npix / 8)
        cfg, wl, imgs = _case(npix, n_sets, 2)
        stacks.append(bioem.prepare_images(ctx, _dev(imgs), cfg.pixel_A))
        shifts.append(shift)
        for m in range(2):
            atoms = wl["atoms"] * np.float32([1.0, 1.0, 1.0 - 0.2 * m, 1.0])
            projsets[m].append(bioem.project_model(ctx, _dev(atoms), cfg.sigma_A, _dev(wl["quats"]), wl["ctfs"], npix, cfg.pixel_A))
            refs[m].append(oracle.score(imgs, atoms, wl["quats"], wl["ctfs"], cfg.sigma_A, cfg.pixel_A, shift)["logP"])
    batch = bioem.Batch(ctx, stacks, projsets, shifts)
    got = batch.run().cpu().numpy()
    batch.close()
    assert ctx.status() == 0
    for m in range(2):
        np.testing.assert_allclose(got[m], np.concatenate(refs[m]), rtol=3e-7, atol=TOL)


@pytest.mark.parametrize("shift", [24, 7])
def test_lists_at_192_px(env, shift):
    """Each image against its own list: the values of the whole range's pairs (1e-9: the pair sums of the two
    calls round ln L in a different order)."""
    import torch
    bioem, ctx = env
    lengths = [3, 0, 1, 40, 0, 5]
    cfg, wl, _ = _case(192, 31, 1)
    rng = np.random.default_rng(192)
    im = bioem.prepare_images(ctx, _dev(rng.standard_normal((6, 192, 192)).astype(np.float32)), cfg.pixel_A)
    ps = bioem.project_model(ctx, _dev(wl["atoms"]), cfg.sigma_A, _dev(wl["quats"]), wl["ctfs"], 192, cfg.pixel_A)
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    idx = rng.integers(0, 31, off[-1]).astype(np.int32)
    got = bioem.score_gathered_pairs(ctx, im, ps, shift, _dev(off), _dev(idx), max(lengths))
    _, plse = bioem.score_pairs(ctx, im, ps, shift)
    want = plse[torch.from_numpy(np.repeat(np.arange(6), lengths)).to(plse.device), _dev(idx).long()]
    assert float((got - want).abs().max()) < 1e-9 and ctx.status() == 0
