"""General absorption where its kernels branch: particles with A on both sides of
1 (the two forms of 1 - exp(-tau)), negative and zero A left out, and tiles cut
into 2, 7, 8, 9 and more segments (the composition takes eighths of them), against the FP64
oracle within the mode's bar (1e-4)."""
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


@pytest.mark.parametrize("tile", [16, 32, 64])
@pytest.mark.parametrize("n,scale", [(900, 1.0), (1500, 2.5), (7100, 0.05), (8300, 1.0), (9300, 0.3)])
def test_one_crowded_tile(rnd, tile, n, scale):
    import torch
    rng = np.random.default_rng(n)
    # every particle reaches the middle tile: lists of n entries, cut every 1024
    p = {"x": rng.normal(0.5, 0.002, n), "y": rng.normal(0.5, 0.002, n), "z": rng.random(n),
         "h": np.exp(rng.uniform(-6.0, -4.5, n)), "I": scale * rng.random(n) ** 4, "s": rng.random(n)}
    p = {k: v.astype(np.float32) for k, v in p.items()}
    cam = scenes.camera(3 * 64, 2 * 64 + 5)
    g = gpu_render(rnd, torch, p, scenes.ramp_palette(), cam, mode=2, tile_px=tile)
    par = {"mode": 2}
    o = oracle.render(p, scenes.ramp_palette(), cam, par, nthreads=os.cpu_count() or 1)
    B, _ = oracle.ambiguity(p, scenes.ramp_palette(), cam, par)
    assert rel_pixel_error(g, o, B) <= 1e-4


# the lists in depth order: one tile (no tile bits), 2^k and 2^k + 1 tiles around the passes of
# up to eight bits, more than 2^16; particles around a warp's run of 32 and its doubling above
# 2^21; depths that are all equal or in a few planes keep the index order
@pytest.mark.parametrize("n,width,height,tile,planes", [
    (1, 16, 16, 16, 1), (33, 64, 64, 64, 4), (500, 256, 256, 16, 1), (511, 272, 256, 16, 3),
    (4097, 512, 520, 32, 0), (3000, 4112, 4096, 16, 5), (65 * 32, 100, 37, 32, 2),
    (2_097_185, 48, 40, 16, 0)])
def test_lists_in_depth_order(rnd, n, width, height, tile, planes):
    import torch
    rng = np.random.default_rng(n)
    h = 1e-4 if n > 10000 else 0.02 if width < 1000 else 0.002
    p = {"x": rng.random(n), "y": rng.random(n), "z": rng.random(n), "h": np.full(n, h),
         "I": np.full(n, 2.0 if n < 10000 else 0.02), "s": rng.random(n)}
    if planes:
        p["z"] = np.floor(p["z"] * planes) / planes
    p = {k: v.astype(np.float32) for k, v in p.items()}
    cam = scenes.camera(width, height)
    g = gpu_render(rnd, torch, p, scenes.ramp_palette(), cam, mode=2, tile_px=tile)
    par = {"mode": 2}
    o = oracle.render(p, scenes.ramp_palette(), cam, par, nthreads=os.cpu_count() or 1)
    B, _ = oracle.ambiguity(p, scenes.ramp_palette(), cam, par)
    assert rel_pixel_error(g, o, B) <= 1e-4


# more segments than are worked on at a time: those behind opaque ones are left out, tile by tile
# (and part by part at 64), those behind transparent ones are not; `right` scales A in the
# right half of the image
@pytest.mark.parametrize("sched", [0, 1])
@pytest.mark.parametrize("tile", [16, 32, 64])
@pytest.mark.parametrize("right", [1.0, 1e-3, 1e-6])
def test_hidden_segments(rnd, tile, right, sched):
    import torch
    n, rng = 620_000, np.random.default_rng(5)
    p = {k: rng.random(n) for k in ("x", "y", "z", "I")}
    p["x"], p["y"] = 2 * p["x"] - 0.5, 2 * p["y"] - 0.5       # the whole image is covered
    p["h"] = rng.uniform(0.01, 0.03, n)
    p["I"] *= np.where(p["x"] > 0.5, right, 1.0)
    p["s"] = rng.random(n)
    p = {k: v.astype(np.float32) for k, v in p.items()}
    pal = scenes.ramp_palette()
    cam = scenes.camera(75, 61)
    g = gpu_render(rnd, torch, p, pal, cam, mode=2, tile_px=tile, sched=sched)
    par = {"mode": 2}
    o = oracle.render(p, pal, cam, par, nthreads=os.cpu_count() or 1)
    B, _ = oracle.ambiguity(p, pal, cam, par)
    assert rnd.stats()["n_entries"][2] > 1024 * (75 * 61 / tile ** 2 + 500)
    assert rel_pixel_error(g, o, B) <= 1e-4
