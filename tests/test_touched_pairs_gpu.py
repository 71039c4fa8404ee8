"""The projection adjoints work only the pairs that the raster backward
touched; the others (hidden behind what ended the pixels before them, or out of
sight) have zero gradients, and the views that see them still count."""
import numpy as np
import pytest

from paper_2510_26358_gb300 import scenes as S
from tests.gpu_helpers import params_to_dev, rel_l2

pytestmark = pytest.mark.gpu

FIELDS = ("means", "log_scales", "quats", "opacity_logits", "sh")


def _scene(n, deg):
    """`n` small Gaussians at z 3..5, the middle third of them behind a wall of
    opaque ones at z 2 (which end every pixel they cover), two equal views."""
    sc = S.random_box_scene(n, 160, 120, 150.0, seed=n, sh_degree=deg, box=((-1.5, 1.5), (-1, 1), (3, 5)),
                            log_scale_mu=-4.0)
    wall = S.random_box_scene(600, 160, 120, 150.0, seed=1, sh_degree=deg, box=((-0.5, 0.5), (-0.5, 0.5), (2, 2.1)),
                              log_scale_mu=-2.0)
    wall.opacity_logits[:] = 4.0
    for k in FIELDS:
        setattr(sc, k, np.concatenate([getattr(sc, k), getattr(wall, k)]))
    sc.submap_offsets = np.array([0, n + 600])
    sc.cameras = sc.cameras * 2
    return sc


# chunk edges of the adjoints (256 Gaussians), and a stretch of Gaussians that
# no view sees, whose rows are cleared in 16-byte pieces
@pytest.mark.parametrize("n", [1, 255, 257, 1500])
@pytest.mark.parametrize("deg", [0, 2, 3])
@pytest.mark.parametrize("unseen", [0, 700])
def test_untouched_rows_are_zero_and_counted(n, deg, unseen):
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    sc = _scene(n, deg)
    if unseen:
        behind = S.random_box_scene(unseen, 160, 120, 150.0, seed=2, sh_degree=deg, box=((-1, 1), (-1, 1), (-5, -2)))
        for k in FIELDS:
            setattr(sc, k, np.concatenate([getattr(behind, k), getattr(sc, k)]))
        sc.submap_offsets = np.array([0, n + 600 + unseen])
    P = params_to_dev(sc)
    r = G.Renderer(sc.cameras, sc.submap_offsets, deg, inst_capacity=1 << 20)
    r.forward(*P)
    gen = torch.Generator(device="cuda").manual_seed(0)
    up = [torch.randn(k, device="cuda", generator=gen) for k in (3 * r.n_pix, r.n_pix)]
    fresh = r.backward(*P, *up)
    g2d = r.buffer(G.BUF_G2D, torch.float32).view(2, -1, 10)
    vis = (r.buffer(G.BUF_PAIR_KEYS, torch.int32) != -1).view(2, -1)
    touched = ((g2d != 0).any(2) & vis).any(0)
    if n == 1500:
        assert (vis.any(0) & ~touched).sum() > 100 and touched.sum() > 100
    assert torch.equal(fresh["densify_cnt"], vis.sum(0, dtype=torch.int32))
    for k in FIELDS + ("densify_acc",):
        assert not fresh[k][~touched].any(), k
        assert torch.isfinite(fresh[k]).all(), k
    # accumulating onto buffers that hold something gives that plus the same
    held = {k: torch.randn(v.shape, device="cuda", generator=gen) if v.is_floating_point() else
            torch.randint(0, 9, v.shape, device="cuda", generator=gen, dtype=v.dtype) for k, v in fresh.items()}
    acc = r.backward(*P, *up, grads={k: v.clone() for k, v in held.items()})
    assert torch.equal(acc["densify_cnt"], held["densify_cnt"] + fresh["densify_cnt"])
    for k in FIELDS + ("densify_acc",):
        assert torch.equal(acc[k][~touched], held[k][~touched]), k
        assert rel_l2((acc[k] - held[k]).cpu(), fresh[k].cpu()) < 1e-4 or not fresh[k].any(), k
    # a later projection forgets what was touched: everything hidden leaves zeros
    P[3] = torch.full_like(P[3], -9.0)
    r.forward(*P)
    none = r.backward(*P, *up)
    for k in FIELDS + ("densify_acc", "densify_cnt", "pose"):
        assert not none[k].any(), k
    r.close()
