"""A tile whose pixels have all ended is left, however few of its remaining
entries reach each quadrant: the forward's time must not grow with what lies
hidden behind a wall."""
import numpy as np
import pytest

from paper_2510_26358_gb300 import scenes as S
from tests.gpu_helpers import params_to_dev

pytestmark = pytest.mark.gpu


def _forward_us(hidden, var):
    """One 32x16 tile, a wall of opaque Gaussians and `hidden` small ones behind
    it, four to each of the tile's eight quadrants in every 32 by depth."""
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    n, f = 4 + hidden, 100.0
    sc = S.random_box_scene(n, 32, 16, f, seed=7)
    i = np.arange(hidden)
    z = 2.0 + 1e-4 * i
    sc.means[:4] = [[0, 0, 1 + 0.01 * k] for k in range(4)]
    sc.log_scales[:4], sc.opacity_logits[:4] = 1.0, 9.0
    u, v = 8 * (i % 4) + 4.0, 8 * (i // 4 % 2) + 4.0
    sc.means[4:] = np.stack([(u - 16) / f * z, (v - 8) / f * z, z], 1)
    sc.log_scales[4:], sc.opacity_logits[4:] = -8.0, 0.0
    r = G.Renderer(sc.cameras, sc.submap_offsets, 0, inst_capacity=1 << 18,
                   config=G.gs_config_default(tile_w=32, tile_h=16, batch_depth=128))
    P = params_to_dev(sc)
    G.gs_workspace_set_profiling(r.ws, True)
    us = []
    for _ in range(6):
        out = r.forward(*P, var=var)
        torch.cuda.synchronize()
        us.append(1e3 * G.gs_workspace_stage_ms(r.ws)["raster_fwd"])
    st, need, seen = r.status()
    assert st == G.GS_OK and seen == n and need >= n
    assert (r.buffer(G.BUF_LAST, torch.int32) <= 4).all() and (out[2] > 0.98).all()
    r.close()
    return min(us)


@pytest.mark.parametrize("var", [False, True])
def test_time_does_not_grow_with_what_is_hidden(var):
    # 60,000 hidden entries are 940 batches of 64, each staged and walked in about a microsecond
    assert _forward_us(60_000, var) < 3 * _forward_us(64, var) + 30
