"""Renderers of sets of different sizes side by side in one process: each from a thread of its
own, and a captured batch replayed after a frame of another size.  Every call succeeds, with
the image that the renderer gives alone (the sums' order is free: 1e-5)."""
import threading

import numpy as np
import pytest

from paper_1309_1114_gb300 import scenes
from tests._metrics import rel_pixel_error

pytestmark = pytest.mark.gpu
# sizes on the three sides of the binning's chunk rule (at 3 and 10 chunks of 2048 per SM)
SIZES = [20_000, 2_000_000, 4_000_000]


@pytest.fixture
def renderers():
    import torch
    from paper_1309_1114_gb300.splotch import Renderer
    made = []
    for n in SIZES:
        sc = scenes.make("uniform", n=n, width=128)
        r = Renderer(0, stream=torch.cuda.Stream().cuda_stream)
        r.load(dict(sc.parts, h=sc.parts["h"] * np.float32(0.05)))
        r.set_colormap(sc.palette)
        r.set_camera(sc.cams[0])
        img = torch.empty((128, 128, 3), device="cuda")
        r.render(img)
        torch.cuda.synchronize()
        made.append((r, sc.cams[0], img.cpu().numpy().astype(np.float64)))
    yield made
    for r, _, _ in made:
        r.close()


def same(img, base):
    M = np.abs(base).reshape(-1, 3).max(0)
    return rel_pixel_error(img.cpu().numpy().astype(np.float64), base, M=M) <= 1e-5


def test_a_thread_each(renderers):
    import torch
    imgs = [torch.empty((128, 128, 3), device="cuda") for _ in renderers]
    stop, failed = threading.Event(), []

    def frames(k):
        r, _, _ = renderers[k]
        try:
            for _ in range(1500):
                if stop.is_set():
                    return
                r.render(imgs[k])
        except Exception as e:      # noqa: BLE001
            failed.append(e)
            stop.set()

    threads = [threading.Thread(target=frames, args=(k,)) for k in range(len(renderers))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed
    for img, (_, _, base) in zip(imgs, renderers):
        assert same(img, base)


def test_a_replay_after_a_frame_of_another_size(renderers):
    import torch
    (small, _, _), (large, cam, base) = renderers[0], renderers[-1]
    imgs = [torch.empty((128, 128, 3), device="cuda") for _ in range(2)]
    other = torch.empty((128, 128, 3), device="cuda")
    for _ in range(3):              # eager, then the graph
        large.render_batch([cam] * 2, imgs)
        small.render(other)
    torch.cuda.synchronize()
    assert same(imgs[0], base) and same(imgs[1], base)
