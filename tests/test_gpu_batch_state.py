"""A batch captured without recording is not replayed once recording is on: every render
stores its own samples then, from the first call and from the replay (features against the
oracle's counts, with the tolerances of the single frame's feature test)."""
import numpy as np
import pytest

import oracle
from paper_1309_1114_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture
def rnd():
    import torch
    assert torch.cuda.is_available()
    from paper_1309_1114_gb300.splotch import Renderer
    r = Renderer(0)
    yield r
    r.close()


def test_recording_switched_on_after_the_capture(rnd):
    import torch
    sc = scenes.make("uniform", n=20_000, width=320)
    cams = [sc.cams[0], scenes.camera(320, azimuth_deg=120.0)]
    imgs = [torch.empty((320, 320, 3), device="cuda") for _ in cams]
    rnd.load(sc.parts)
    rnd.set_colormap(sc.palette)
    rnd.set_params(r_small=4.0, r_large=1e9)        # no large class, and no tile is cut
    for _ in range(2):
        rnd.render_batch(cams, imgs)                # captured and replayed
    ref = np.concatenate([oracle.tile_features(sc.parts, sc.palette, c, {}, 32, area_scale=1024) for c in cams])
    ref = ref[ref[:, :16].sum(1) > 0]
    rnd.set_recording(True)
    f, t = torch.empty((4096, 32), device="cuda"), torch.empty(4096, device="cuda")
    for _ in range(2):
        rnd.render_batch(cams, imgs)
        f.zero_(), t.zero_()
        torch.cuda.synchronize()
        n = rnd.samples(f, t)
        got = f[:n].cpu().numpy().astype(np.float64)
        assert got.shape == ref.shape
        cg, cr = np.expm1(got[:, :16]), np.expm1(ref[:, :16])
        assert np.abs(cg - cr).sum() <= 2 * len(cams) + 0.002 * cr.sum()
        assert np.mean(np.abs(got - ref) < 1e-4) > 0.99
        assert t[:n].min().item() > 0
