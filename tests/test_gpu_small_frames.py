"""Small frames, whose list segments shrink: every size class around the shortened
segments, one view and a batch, each tile side, against the FP64 oracle within the
FP32 bar (1e-4); the recorded samples keep the full segments."""
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


def crowded(n, seed):
    """n particles in and around one tile: points, small, medium and large."""
    rng = np.random.default_rng(seed)
    p = {"x": rng.normal(0.5, 0.02, n), "y": rng.normal(0.5, 0.02, n), "z": rng.random(n),
         "h": np.exp(rng.uniform(-9.0, -2.0, n)), "I": rng.random(n), "s": rng.random(n)}
    return {k: v.astype(np.float32) for k, v in p.items()}


@pytest.mark.parametrize("tile", [16, 32, 64])
@pytest.mark.parametrize("n", [100, 129, 300, 1100, 5000])
def test_shortened_segments(rnd, tile, n):
    import torch
    p, cam = crowded(n, n), scenes.camera(100, 90)
    pal = scenes.ramp_palette()
    o = oracle.render(p, pal, cam, {}, nthreads=os.cpu_count() or 1)
    B, _ = oracle.ambiguity(p, pal, cam, {})
    g = gpu_render(rnd, torch, p, pal, cam, tile_px=tile, r_large=12.0)
    assert rel_pixel_error(g, o, B) <= 1e-4
    imgs = [torch.empty((90, 100, 3), device="cuda") for _ in range(3)]
    for _ in range(2):                       # eager, then the graph
        rnd.render_batch([cam] * 3, imgs)
        torch.cuda.synchronize()
        for im in imgs:
            assert rel_pixel_error(im.cpu().numpy().astype(np.float64), o, B) <= 1e-4


def test_recorded_items_keep_full_segments(rnd):
    import torch
    p, cam = crowded(900, 1), scenes.camera(64, 64)
    rnd.set_recording(True)
    try:
        gpu_render(rnd, torch, p, scenes.ramp_palette(), cam, r_large=1e6)
        feat, logc = torch.empty((4096, 32), device="cuda"), torch.empty(4096, device="cuda")
        n = rnd.samples(feat, logc)
    finally:
        rnd.set_recording(False)
    # 900 entries per tile at most: one item each
    assert n == 4


@pytest.mark.parametrize("grow", [4.0, 40.0])
def test_replayed_lists_that_outgrow_their_buffers(grow):
    """The passes of a replayed graph must not read entries past the buffer their lists
    outgrew (a fresh context: nothing larger was rendered in it before)."""
    import torch
    from paper_1309_1114_gb300.splotch import Renderer
    p = scenes.make("uniform", n=30_000).parts
    big = dict(p, h=(p["h"] * np.float32(grow)))
    cams = [scenes.camera(160, 120, azimuth_deg=a) for a in (0.0, 120.0)]
    r = Renderer(0)
    try:
        r.set_colormap(scenes.ramp_palette())
        r.set_params(r_large=20.0)
        imgs = [torch.empty((120, 160, 3), device="cuda") for _ in cams]
        for parts in (p, p, big):            # eager, replay, a replay that overflows
            r.load(parts)
            r.render_batch(cams, imgs)
        torch.cuda.synchronize()
        for cam, im in zip(cams, imgs):
            o = oracle.render(big, scenes.ramp_palette(), cam, {}, nthreads=os.cpu_count() or 1)
            B, _ = oracle.ambiguity(big, scenes.ramp_palette(), cam, {})
            assert rel_pixel_error(im.cpu().numpy().astype(np.float64), o, B) <= 1e-4
    finally:
        r.close()


@pytest.mark.parametrize("chunks", [3, 10])      # 2048-particle chunks per SM where the binning
@pytest.mark.parametrize("off", [-1, 0])         # goes from quarter to half chunks, and to whole ones
def test_chunk_sizes_meet(rnd, chunks, off):
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count * chunks * 2048 + off
    rng = np.random.default_rng(chunks)
    p = {k: rng.random(n, dtype=np.float32) for k in ("x", "y", "z", "I", "s")}
    p["h"] = np.exp(rng.uniform(-9.0, -6.0, n)).astype(np.float32)
    pal, cam = scenes.ramp_palette(), scenes.camera(400, 300)
    o = oracle.render(p, pal, cam, {}, nthreads=os.cpu_count() or 1)
    B, _ = oracle.ambiguity(p, pal, cam, {})
    g = gpu_render(rnd, torch, p, pal, cam, tile_px=16)
    assert rel_pixel_error(g, o, B) <= 1e-4
