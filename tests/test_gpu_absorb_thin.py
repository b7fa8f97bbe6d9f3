"""General absorption: the error of one particle's 1 - exp(-tau) for A <= 1, and its mean, which a
sum over many thin particles would add up.  One point per pixel (weight 1, tau = A): the
image is E / A (1 - exp(-A)), with five roundings: E, 1 / A, their product, 1 - exp(-A), the
result.  Each is at most 2^-24 relative and 2^-24 / sqrt(3) rms, together 7.7e-8 rms, so that
the mean over 4096 pixels has a standard error of 1.2e-9: within 1e-8 of zero."""
import numpy as np
import pytest

from paper_1309_1114_gb300 import scenes
from tests.test_gpu_parity import gpu_render
from tests.test_gpu_tile_edges import at_pixels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(1e-7, 1e-4), (1e-4, 1e-2), (1e-2, 1 / 16), (1 / 16, 1 / 8), (1 / 8, 1 / 2), (1 / 2, 1.0)])
def test_no_bias_of_one_particle(lo, hi):
    import torch
    from paper_1309_1114_gb300.splotch import Renderer
    w, rng = 64, np.random.default_rng(3)
    cam = scenes.camera(w, w)
    gx, gy = np.meshgrid(np.arange(w) + 0.5, np.arange(w) + 0.5)
    p = at_pixels(gx.ravel(), gy.ravel(), np.full(w * w, 0.1), cam, rng)
    p["I"] = np.exp(rng.uniform(np.log(lo), np.log(hi), w * w))
    for k in ("cr", "cg", "cb"):
        p[k] = rng.uniform(0.5, 1.0, w * w)
    p = {k: np.asarray(v, np.float32) for k, v in p.items()}
    r = Renderer(0)
    try:
        g = gpu_render(r, torch, p, scenes.ramp_palette(), cam, mode=2)
    finally:
        r.close()
    gain = -np.expm1(-p["I"].astype(np.float64)).reshape(w, w, 1)
    want = gain * np.stack([p[k].astype(np.float64) for k in ("cr", "cg", "cb")], 1).reshape(w, w, 3)
    err = g / want - 1.0
    assert np.abs(err).max() <= 5 * 2.0 ** -23
    assert np.sqrt((err ** 2).mean()) <= 7.7e-8 and abs(err.mean()) <= 1e-8
