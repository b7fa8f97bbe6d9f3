"""The covering pass of large particles (tiles wholly inside a disc): every number of
covering entries around its batches and its threshold, discs that just cover or
just miss covering a tile, tile sides 32 and 64, ragged images, a batch, a long list cut
into several items, against the FP64 oracle within the FP32 bar (1e-4)."""
import os

import numpy as np
import pytest

import oracle
from paper_1309_1114_gb300 import scenes
from tests._metrics import rel_pixel_error
from tests.test_gpu_parity import gpu_render
from tests.test_gpu_tile_edges import at_pixels

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rnd():
    import torch
    assert torch.cuda.is_available()
    from paper_1309_1114_gb300.splotch import Renderer
    r = Renderer(0)
    yield r
    r.close()


def reference(p, cam):
    o = oracle.render(p, scenes.ramp_palette(), cam, {}, nthreads=os.cpu_count() or 1)
    B, _ = oracle.ambiguity(p, scenes.ramp_palette(), cam, {})
    return o, B


@pytest.mark.parametrize("tile", [16, 32, 64])
@pytest.mark.parametrize("n", [63, 64, 65, 127, 129, 191, 513, 2500])
def test_numbers_of_covering_entries(rnd, tile, n):
    import torch
    rng = np.random.default_rng(n)
    cam = scenes.camera(75, 70)
    p = at_pixels(rng.uniform(-40, 110, n), rng.uniform(-40, 110, n), rng.uniform(70, 400, n), cam, rng)
    p = {k: np.asarray(v, np.float32) for k, v in p.items()}
    o, B = reference(p, cam)
    g = gpu_render(rnd, torch, p, scenes.ramp_palette(), cam, tile_px=tile)
    assert rel_pixel_error(g, o, B) <= 1e-4
    imgs = [torch.empty((70, 75, 3), device="cuda") for _ in range(2)]
    for _ in range(2):                       # eager, then the graph
        rnd.render_batch([cam] * 2, imgs)
    torch.cuda.synchronize()
    assert rel_pixel_error(imgs[1].cpu().numpy().astype(np.float64), o, B) <= 1e-4


@pytest.mark.parametrize("tile", [32, 64])
def test_discs_that_just_cover_a_tile(rnd, tile):
    import torch
    rng = np.random.default_rng(tile)
    cam = scenes.camera(2 * tile, tile)
    # the farthest pixel centre of the left tile, seen from its middle
    far = np.hypot(0.5 * tile - 0.5, 0.5 * tile - 0.5)
    n = 200
    r = far * (1.0 + np.repeat([-1e-3, -1e-5, -1e-6, 0.0, 1e-6, 1e-5, 1e-3, 0.1], n // 8))
    p = at_pixels(0.5 * tile + np.zeros(n), 0.5 * tile + np.zeros(n), r, cam, rng)
    p = {k: np.asarray(v, np.float32) for k, v in p.items()}
    o, B = reference(p, cam)
    g = gpu_render(rnd, torch, p, scenes.ramp_palette(), cam, tile_px=tile, r_large=10.0)
    assert rel_pixel_error(g, o, B) <= 1e-4
