"""The covering pass inside its items: full and partial batches of 64, several of them, items that
cover their tile with a part of their entries only, sole and cut large lists, long segments, and
discs on either side of covering a tile, enough of each that an item takes the pass or does
not.  Against the FP64 oracle within the FP32 bar (1e-4)."""
import os

import numpy as np
import pytest

import oracle
from paper_1309_1114_gb300 import scenes
from tests._metrics import rel_pixel_error
from tests.test_gpu_parity import gpu_render
from tests.test_gpu_tile_edges import at_pixels

pytestmark = pytest.mark.gpu
R_LARGE = 8.0


@pytest.fixture(scope="module")
def rnd():
    import torch
    assert torch.cuda.is_available()
    from paper_1309_1114_gb300.splotch import Renderer
    r = Renderer(0)
    yield r
    r.close()


def covers(px, py, r, x0, y0, x1, y1):
    """Does the disc take the covering pass on the tile of pixels [x0, x1) x [y0, y1)?"""
    dx = np.maximum(px - (x0 + 0.5), (x1 - 0.5) - px)
    dy = np.maximum(py - (y0 + 0.5), (y1 - 0.5) - py)
    return np.hypot(dx, dy) <= r - 1e-3 - 4e-6 * r


def check(rnd, torch, px, py, r, cam, tile, sched, batch=False):
    rng = np.random.default_rng(len(px))
    p = at_pixels(px, py, r, cam, rng)
    p = {k: np.asarray(v, np.float32) for k, v in p.items()}
    pal = scenes.ramp_palette()
    o = oracle.render(p, pal, cam, {}, nthreads=os.cpu_count() or 1)
    B, _ = oracle.ambiguity(p, pal, cam, {})
    imgs = [gpu_render(rnd, torch, p, pal, cam, tile_px=tile, r_large=R_LARGE, sched=sched)]
    n_large = rnd.stats()["n_entries"][3]
    tiles = -(-cam["width"] // tile) * -(-cam["height"] // tile)
    assert n_large >= 64 * tiles or len(px) < 64    # the frame has a covering pass
    if batch:
        out = [torch.empty((cam["height"], cam["width"], 3), device="cuda") for _ in range(2)]
        for _ in range(2):                          # eager, then the graph
            rnd.render_batch([cam] * 2, out)
        torch.cuda.synchronize()
        imgs += [im.cpu().numpy().astype(np.float64) for im in out]
    for g in imgs:
        assert rel_pixel_error(g, o, B) <= 1e-4
    return n_large


# with a schedule, large lists are cut every 512 entries whatever the frame's size; the
# covering entries come last.  n_part = 600: the first item has none, the second the rest
@pytest.mark.parametrize("tile", [32, 64])
@pytest.mark.parametrize("n_part", [0, 3, 150, 600])
@pytest.mark.parametrize("n_cover", [63, 64, 65, 67, 127, 128, 129, 130, 191, 320, 421])
def test_covering_entries_of_an_item(rnd, tile, n_part, n_cover):
    import torch
    rng = np.random.default_rng(1000 * n_part + n_cover)
    # a whole tile and a ragged one beside it
    cam = scenes.camera(tile + 11, tile - 3)
    n = n_part + n_cover
    px, py = rng.uniform(0.0, tile, n), rng.uniform(0.0, tile, n)
    r = rng.uniform(2.0, 5.0, n) * tile
    r[:n_part] = rng.uniform(R_LARGE + 1.0, 0.49 * tile, n_part)
    order = rng.permutation(n)
    full = covers(px, py, r, 0, 0, tile, tile - 3)
    assert full[n_part:].all() and not full[:n_part].any()
    check(rnd, torch, px[order], py[order], r[order], cam, tile, 1, batch=n_part == 150)


# without one they are cut to the frame: 8 items per SM, at least 64 entries each
@pytest.mark.parametrize("tile,width,n", [(32, 64, 100_000), (64, 64, 200_000)])
def test_long_segments(rnd, tile, width, n):
    import torch
    rng = np.random.default_rng(n)
    cam = scenes.camera(width, tile)
    px, py = rng.uniform(0.0, width, n), rng.uniform(0.0, tile, n)
    r = rng.uniform(R_LARGE + 1.0, 300.0, n)
    share = covers(px, py, r, 0, 0, tile, tile).mean()
    assert 0.5 < share < 0.95
    n_large = check(rnd, torch, px, py, r, cam, tile, 0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert n_large // (8 * sms) > 128               # three batches and more


# one radius at a time: all discs of an item cover the tile, or none.  (far: the corner pixels'
# centres, seen from the tile's middle)
@pytest.mark.parametrize("tile", [32, 64])
@pytest.mark.parametrize("off", [-1e-3, -1e-4, -1e-5, -1e-6, 0.0, 1e-6, 1e-5, 1e-4, 1e-3, 0.1])
def test_discs_of_one_radius(rnd, tile, off):
    import torch
    cam = scenes.camera(tile, tile)
    n, mid = 300, np.full(300, 0.5 * tile)
    far = np.hypot(0.5 * tile - 0.5, 0.5 * tile - 0.5)
    r = np.full(n, far * (1.0 + off))
    edge = r * (1.0 - 4e-6) - 1e-3 - far
    assert (np.abs(edge) > 2e-5).all()              # FP32 cannot decide otherwise
    assert covers(mid, mid, r, 0, 0, tile, tile).all() == (off >= 1e-4)
    assert check(rnd, torch, mid, mid, r, cam, tile, 1) == n
