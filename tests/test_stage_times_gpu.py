"""With profiling on, every stage that a call runs reads a time, also where
another stage's kernel takes its work along."""
import pytest

from paper_2510_26358_gb300 import scenes as S
from tests.gpu_helpers import params_to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1000, 20_000])  # one launch for compaction and depth sort up to 16,384 pairs
@pytest.mark.parametrize("lam", [0.0, 0.2])    # the L1 term in the SSIM kernels unless lambda is 0
def test_every_stage_reads_a_time(n, lam):
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    sc = S.random_box_scene(n, 161, 119, 150.0, seed=4)
    P = params_to_dev(sc)
    r = G.Renderer(sc.cameras, sc.submap_offsets, 0, inst_capacity=1 << 20)
    G.gs_workspace_set_profiling(r.ws, True)
    rgb, depth, alpha = r.forward(*P)
    g = torch.zeros_like(rgb)
    r.image_loss(rgb, torch.rand_like(rgb), lam, g)
    r.backward(*P, g, torch.zeros_like(depth))
    ms = G.gs_workspace_stage_ms(r.ws)
    want = set(G.STAGES) - {"depth_loss", "zero_grad"}
    assert set(ms) >= want and all(ms[k] < 100 for k in want)
    r.close()
