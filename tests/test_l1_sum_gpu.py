"""The L1 term of gs_image_loss is the correctly rounded mean where every sum
that leads to it can be: of four row values whose plain float sum is two ulps
off.  64x64 stages by TMA, 63x64 by plain loads."""
import numpy as np
import pytest

from paper_2510_26358_gb300 import scenes as S

pytestmark = pytest.mark.gpu

ROWS = np.array([1033305520, 1064904749, 1058184839, 1051460574], np.uint32).view(np.float32)


@pytest.mark.parametrize("width", [64, 63])
@pytest.mark.parametrize("lam", [0.2, 1.0])
def test_l1_is_the_rounded_mean(width, lam):
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    plain = np.float32(0)
    for x in ROWS:
        plain += x
    want = np.float32(ROWS.astype(np.float64).mean())
    assert np.float32(plain / 4) != want  # (a division by four is exact)
    sc = S.random_box_scene(1, width, 64, 60.0, seed=0)
    r = G.Renderer(sc.cameras, sc.submap_offsets, 0, inst_capacity=1 << 16)
    x = torch.from_numpy(np.tile(np.repeat(ROWS, width), 3 * 64 // 4)).cuda()
    loss = r.image_loss(x, torch.zeros_like(x), lam, torch.zeros_like(x)).cpu().numpy()
    assert loss[1] == want
    # a value that is not finite is not hidden
    x[70] = float("inf")
    assert np.isinf(r.image_loss(x, torch.zeros_like(x), lam, torch.zeros_like(x)).cpu().numpy()[1])
    r.close()
