"""Codes of the 16-bit logarithmic smoothing length where FP32 cannot decide
them: h a few ulps around half steps, at the clamps, subnormal, huge, with
h_log2_min values that are not exact in binary.  The codes must equal the FP64
definition, except where numpy's own FP64 value lies within 1e-9 of a half step."""
import numpy as np
import pytest

from paper_1309_1114_gb300 import splotch as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h_log2_min", [-14.0, -13.987654, -3.3, 0.1, -126.7, 100.25, 3.0e38])
def test_codes_at_half_steps_and_clamps(h_log2_min):
    import torch
    rng = np.random.default_rng(5)
    lo = np.float64(np.float32(h_log2_min))
    k = rng.integers(0, 65535, 60000)
    with np.errstate(over="ignore"):
        h = np.exp2(lo + (k + 0.5) / 4096.0).astype(np.float32)
        h = np.concatenate([h, np.nextafter(h, np.float32(0)), np.nextafter(h, np.float32(np.inf)),
                            np.exp2(rng.uniform(-149, 127, 20000)).astype(np.float32),
                            np.exp2(lo + rng.uniform(-0.01, 0.01, 500)).astype(np.float32),
                            np.exp2(lo + 16 + rng.uniform(-0.01, 0.01, 500)).astype(np.float32)])
    h = h[np.isfinite(h) & (h > 0)]
    t = (np.log2(h.astype(np.float64)) - lo) * 4096.0
    want = np.clip(np.rint(t), 0, 65535).astype(np.int64)
    sure = np.abs(np.abs(t - np.floor(t)) - 0.5) > 1e-9
    r = S.Renderer(0)
    d = torch.from_numpy(h).cuda()
    out = r.encode_attrs(d, d, d, S.SPL_ATTR_LOGH16, h_log2_min)
    torch.cuda.synchronize()
    got = out["h"].cpu().numpy().view(np.uint16).astype(np.int64)
    r.close()
    assert sure.mean() > 0.99 and np.array_equal(got[sure], want[sure])
