"""GPU: callers on several host threads, each with its own context and stream."""
import threading

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
    return bioem


def test_proposals_of_different_length_at_once(env):
    """One thread asks for 16,384 bins, another for 1, many times over: neither refuses a call of the other
    (the sorting kernel's shared memory differs by a factor of 256), and both get what one thread gets."""
    import torch
    bioem = env
    errors, done = [], threading.Event()

    def caller(k, stream):
        try:
            with torch.cuda.stream(stream):
                ctx = bioem.Context(0, stream)
                net = bioem.CNN(ctx, image_px=16, downsample=2, channels=4, n_qbins=4608, n_dbins=4, max_batch=4, seed=5)
                gen = torch.Generator(device="cuda:0").manual_seed(1)
                imgs = torch.randn((2, 16, 16), generator=gen, device="cuda:0")
                want = net.propose(imgs, k)
                start.wait(60)
                for _ in range(400):
                    if done.is_set():
                        break
                    got = net.propose(imgs, k)
                    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
                net.close()
        except Exception as e:
            errors.append((k, e))
            done.set()
            start.abort()

    start = threading.Barrier(2)
    threads = [threading.Thread(target=caller, args=(k, torch.cuda.Stream())) for k in (16384, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
