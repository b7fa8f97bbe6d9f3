"""The tile pass at the edges of its batches (64 particles), of its 8 x 8
blocks and of the image: list lengths around a batch and a work item, discs that
just reach or miss a block, ragged image sides, against the FP64 oracle within
the FP32 bar (1e-4)."""
import os

import numpy as np
import pytest

import oracle
from paper_1309_1114_gb300 import scenes
from tests._metrics import rel_pixel_error
from tests.test_gpu_parity import gpu_render

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rnd():
    import torch
    assert torch.cuda.is_available()
    from paper_1309_1114_gb300.splotch import Renderer
    r = Renderer(0)
    yield r
    r.close()


def check(rnd, p, cam, **par):
    import torch
    p = {k: np.asarray(v, np.float32) for k, v in p.items()}
    g = gpu_render(rnd, torch, p, scenes.ramp_palette(), cam, **par)
    op = {k: v for k, v in par.items() if k in ("mode", "chi")}
    o = oracle.render(p, scenes.ramp_palette(), cam, op, nthreads=os.cpu_count() or 1)
    B, _ = oracle.ambiguity(p, scenes.ramp_palette(), cam, op)
    assert np.isfinite(g).all() and rel_pixel_error(g, o, B) <= 1e-4


def at_pixels(px, py, r, cam, rng):
    """Particles at depth 2 with screen position (px, py) and radius r."""
    f = 0.5 * cam["height"] / np.tan(np.radians(30.0))
    n = len(px)
    # the camera looks along +z: screen x runs along -x of the scene
    x = 0.5 - (np.asarray(px) - 0.5 * cam["width"]) * 2.0 / f
    y = 0.5 - (np.asarray(py) - 0.5 * cam["height"]) * 2.0 / f
    return {"x": x, "y": y, "z": np.full(n, 0.5), "h": np.asarray(r) * 2.0 / (3.0 * f),
            "I": rng.random(n), "s": rng.random(n)}


@pytest.mark.parametrize("tile", [16, 32, 64])
@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 127, 128, 129, 1023, 1024, 1025, 2100])
def test_list_lengths(rnd, n, tile):
    rng = np.random.default_rng(n)
    cam = scenes.camera(96, 64)
    p = at_pixels(rng.uniform(33, 63, n), rng.uniform(1, 31, n), rng.uniform(2.1, 12.0, n), cam, rng)
    check(rnd, p, cam, tile_px=tile)


@pytest.mark.parametrize("tile", [16, 32, 64])
@pytest.mark.parametrize("w,h", [(1, 1), (7, 33), (33, 31), (40, 41), (65, 97)])
def test_discs_at_block_edges_of_ragged_images(rnd, w, h, tile):
    rng = np.random.default_rng(w * 100 + h)
    cam = scenes.camera(w, h)
    gx, gy = np.meshgrid(np.arange(-8, w + 9, 8), np.arange(-8, h + 9, 8))
    n = gx.size
    px, py = gx.ravel() + rng.normal(0, 0.02, n), gy.ravel() + rng.normal(0, 0.02, n)
    for r in (0.3, 1.5, 2.05, 3.5, 7.99, 8.01, 30.0):
        check(rnd, at_pixels(px, py, np.full(n, r), cam, rng), cam, tile_px=tile)
    check(rnd, at_pixels(px, py, rng.uniform(0.2, 80.0, n), cam, rng), cam, mode=1, r_large=20.0,
          tile_px=tile)
