"""Renderers open side by side: what a second one needs (another image size or
batch depth takes the same kernels with other launch shapes) must not limit the
first."""
import pytest

from paper_2510_26358_gb300 import scenes as S
from tests.gpu_helpers import params_to_dev, rel_l2

pytestmark = pytest.mark.gpu

GRADS = ("means", "log_scales", "quats", "opacity_logits", "sh", "pose")


def _open(size, tile, depth):
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    sc = S.random_box_scene(2000, *size, 300.0, seed=5)
    r = G.Renderer(sc.cameras, sc.submap_offsets, 0, inst_capacity=1 << 20,
                   config=G.gs_config_default(tile_w=tile[0], tile_h=tile[1], batch_depth=depth))
    gen = torch.Generator(device="cuda").manual_seed(6)
    up = [torch.randn(k * r.n_pix, device="cuda", generator=gen) for k in (3, 1)]
    return r, params_to_dev(sc), up


def _pass(r, P, up, var):
    out = r.forward(*P, var=var)
    extra = dict(dL_dmean=up[1], dL_dvar=up[1]) if var else {}
    g = r.backward(*P, *up, var=var, **extra)
    return [x.cpu().numpy() for x in out], {k: g[k].cpu().numpy() for k in GRADS}


# (size, batch depth) of the first renderer and of the one opened after it:
# 320x240 is 300 tiles of 16x16, 640x480 1200, 1280x960 4800
@pytest.mark.parametrize("first,second", [(((320, 240), 256), ((640, 480), 256)), (((320, 240), 128), ((320, 240), 64)),
                                          (((640, 480), 256), ((320, 240), 32)), (((1280, 960), 256), ((1280, 960), 32))])
@pytest.mark.parametrize("tile", [(8, 8), (16, 16), (16, 32), (32, 16)])
def test_the_first_still_runs(first, second, tile):
    for var in (False, True):
        r, P, up = _open(first[0], tile, first[1])
        images, grads = _pass(r, P, up, var)
        other, Q, dn = _open(second[0], tile, second[1])
        again, g = _pass(r, P, up, var)
        _pass(other, Q, dn, var)
        for a, b in zip(images, again):
            assert (a == b).all()
        for k in GRADS:  # float atomics in another order
            assert rel_l2(g[k], grads[k]) < 1e-5, k
        r.close()
        other.close()
