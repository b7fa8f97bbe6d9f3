"""General absorption with the network scheduler and with recording on, from the first frame
of a context: the item features read the tile lists, which this mode writes in depth order.
The features are compared with the oracle's count per tile (the tolerances of the additive
mode's feature test), the image with the FP64 oracle (1e-4)."""
import os

import numpy as np
import pytest

import oracle
from paper_1309_1114_gb300 import scenes, scheduler
from tests._metrics import rel_pixel_error
from tests.test_gpu_parity import gpu_render

pytestmark = pytest.mark.gpu

# two frames of one context, the second with longer lists, so that the buffers grow in between
SETS = [("uniform", 4_000, 320), ("uniform", 12_000, 320)]


@pytest.mark.parametrize("tile", [16, 32, 64])
def test_recorded_features_are_of_this_frame(tile):
    import torch
    from paper_1309_1114_gb300.splotch import Renderer
    r = Renderer(0)
    try:
        r.set_recording(True)
        for name, n, width in SETS[:1 if tile == 64 else 2]:    # (no tile is cut)
            sc = scenes.make(name, n=n, width=width)
            cam = sc.cams[0]
            gpu_render(r, torch, sc.parts, sc.palette, cam, mode=2, tile_px=tile)
            f, t = torch.empty((4096, 32), device="cuda"), torch.empty(4096, device="cuda")
            n_items = r.samples(f, t)
            ref = oracle.tile_features(sc.parts, sc.palette, cam, {}, tile, area_scale=tile * tile)
            ref = ref[ref[:, :16].sum(1) > 0]
            got = f[:n_items].cpu().numpy().astype(np.float64)
            assert got.shape == ref.shape
            cg, cr = np.expm1(got[:, :16]), np.expm1(ref[:, :16])
            ag, ar = np.expm1(got[:, 16:]) * tile ** 2, np.expm1(ref[:, 16:]) * tile ** 2
            assert np.abs(cg - cr).sum() <= 2 + 0.002 * cr.sum()
            assert np.abs(ag - ar).sum() <= 0.002 * ar.sum()
            assert np.mean(np.abs(got - ref) < 1e-4) > 0.99
    finally:
        r.close()


@pytest.mark.parametrize("recording", [False, True])
@pytest.mark.parametrize("tile", [16, 32, 64])
def test_network_schedule(tile, recording):
    import torch
    from paper_1309_1114_gb300.splotch import Renderer
    r = Renderer(0)
    try:
        r.set_model(scheduler.init_theta(7, bias=10.0))
        r.set_recording(recording)
        for name, n, width in SETS + [("clustered", 100_000, 200)]:      # (cut tiles)
            sc = scenes.make(name, n=n, width=width)
            cam, par = sc.cams[0], {"mode": 2}
            g = gpu_render(r, torch, sc.parts, sc.palette, cam, mode=2, tile_px=tile, sched=2)
            o = oracle.render(sc.parts, sc.palette, cam, par, nthreads=os.cpu_count() or 1)
            B, _ = oracle.ambiguity(sc.parts, sc.palette, cam, par)
            assert rel_pixel_error(g, o, B) <= 1e-4
    finally:
        r.close()
