"""Gradient kernel at the edges of its sample tiles (64 samples, 152 CTAs): one
sample, a tile and one more or less, a partly filled last round of tiles.
Tolerance: FP32 sums of at most 10^4 terms against FP64, 10^-5 of the largest
component (the bar of the other gradient test)."""
import numpy as np
import pytest

import oracle
from paper_1309_1114_gb300 import scheduler
from paper_1309_1114_gb300 import splotch as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 31, 63, 64, 65, 128, 64 * 152, 64 * 152 + 1])
def test_gradient_at_tile_edges(batch):
    import torch
    rng = np.random.default_rng(batch)
    theta = scheduler.init_theta(3, bias=1.0)
    x = rng.uniform(0.0, 6.0, (batch, 32)).astype(np.float32)
    t = rng.uniform(8.0, 14.0, batch).astype(np.float32)
    dev = [torch.from_numpy(a).cuda() for a in (theta, x, t)]
    grad = torch.full((S.SPL_MLP_NPARAM,), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), device="cuda")
    for _ in range(2):      # the second call reuses the scratch
        S.check(S.spl_mlp_loss_grad(dev[0].data_ptr(), dev[1].data_ptr(), dev[2].data_ptr(), batch,
                                    grad.data_ptr(), loss.data_ptr(), None), "spl_mlp_loss_grad")
        l64, g64 = oracle.mlp_loss_grad(theta, x, t)
        assert abs(float(loss) - l64) <= 1e-5 * abs(l64)
        assert np.max(np.abs(grad.cpu().numpy() - g64)) <= 1e-5 * np.max(np.abs(g64))
