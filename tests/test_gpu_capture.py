"""GPU: scoring calls recorded in a CUDA graph after calls of other shapes have sized the scratch memory."""
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
    return bioem


def test_capture_of_fewer_images_and_more_sets(env):
    """64 images x 1024 sets first; then 8 images x 8192 sets, the same records but a reduction in many parts per
    image, are captured: no scratch may grow, and replays on the captured inputs give the eager call's values."""
    import torch
    bioem = env
    cfg = workloads.get_config("tiny", npix=32, pixel_A=2.0, max_shift=4, n_orient=1024, n_defocus=1, bfactors=(0.0,), n_atoms=60)
    wl = workloads.workload(cfg, n_img=1)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        ctx = bioem.Context(0, side)
        gen = torch.Generator(device="cuda:0").manual_seed(2)
        imgs = torch.randn((64, 32, 32), generator=gen, device="cuda:0")
        many = bioem.prepare_images(ctx, imgs, cfg.pixel_A)
        few = bioem.prepare_images(ctx, imgs[:8], cfg.pixel_A)
        quats, atoms = dev(wl["quats"]), dev(wl["atoms"])
        short = bioem.project_model(ctx, atoms, cfg.sigma_A, quats, wl["ctfs"], 32, cfg.pixel_A)
        ctfs = [(5000.0 + 2000.0 * i, 0.1, 0.0, 300.0) for i in range(8)]
        long = bioem.project_model(ctx, atoms, cfg.sigma_A, quats, ctfs, 32, cfg.pixel_A)
        bioem.score(ctx, many, short, 4)
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            out = bioem.score(ctx, few, long, 4)
        for _ in range(2):
            out.zero_()
            graph.replay()
        side.synchronize()
        got = out.clone()
        want = bioem.score(ctx, few, long, 4)
        assert ctx.status() == 0
        assert torch.equal(got, want)
