"""General absorption with particles of A <= 0 (negative intensities, or logarithms of
intensities below 1): they neither emit nor absorb, however many of them a pixel's list holds
behind opaque or transparent particles, in one item or in several, against the FP64 oracle
within the mode's bar (1e-4)."""
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


def check(rnd, p, tile, **par):
    import torch
    p = {k: np.asarray(v, np.float32) for k, v in p.items()}
    # odd sides: the particles, on the optical axis, lie in the middle of a pixel
    cam, pal = scenes.camera(75, 61), scenes.ramp_palette()
    g = gpu_render(rnd, torch, p, pal, cam, mode=2, tile_px=tile, **par)
    q = {"mode": 2, "log": par.get("log_flags", 0)}
    o = oracle.render(p, pal, cam, q, nthreads=os.cpu_count() or 1)
    B, _ = oracle.ambiguity(p, pal, cam, q)
    assert np.isfinite(g).all() and o.max() > 0
    assert rel_pixel_error(g, o, B) <= 1e-4


def on_axis(n, h, rng):
    return {"x": np.full(n, 0.5), "y": np.full(n, 0.5), "z": rng.random(n), "h": np.full(n, h), "s": rng.random(n)}


# one item (up to 1024 entries) and several, some of them with A <= 0 only
@pytest.mark.parametrize("tile", [16, 32, 64])
@pytest.mark.parametrize("h", [1e-5, 0.05])                 # points, discs
@pytest.mark.parametrize("n_pos,n_neg", [(500, 500), (2000, 3000)])
@pytest.mark.parametrize("scale", [1.0, 1e-3])              # opaque, transparent
def test_negative_and_zero_intensities(rnd, tile, h, n_pos, n_neg, scale):
    rng = np.random.default_rng(n_pos)
    p = on_axis(n_pos + n_neg + 24, h, rng)
    p["I"] = rng.permutation(np.concatenate([np.full(n_pos, scale), np.full(n_neg, -1.0), np.zeros(24)]))
    check(rnd, p, tile)


@pytest.mark.parametrize("tile", [16, 32, 64])
@pytest.mark.parametrize("n", [1000, 5000])
def test_logarithms_of_intensities_below_one(rnd, tile, n):
    rng = np.random.default_rng(n)
    p = on_axis(n, 0.05, rng)
    p["I"] = 10.0 ** rng.uniform(-2.0, 1.0, n)
    check(rnd, p, tile, log_flags=1)
