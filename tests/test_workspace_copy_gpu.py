"""gs_workspace_copy copies bytes: any destination will do, whatever its
alignment.  The workspace's memory is what its documented rows take."""
import ctypes

import pytest

from paper_2510_26358_gb300 import scenes as S
from tests.gpu_helpers import params_to_dev

pytestmark = pytest.mark.gpu


def test_every_buffer_copies_to_an_odd_address():
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    sc = S.random_box_scene(500, 161, 119, 150.0, seed=3, sh_degree=1)
    P = params_to_dev(sc)
    r = G.Renderer(sc.cameras, sc.submap_offsets, 1, inst_capacity=1 << 18)
    r.forward(*P, var=True)
    up = [torch.randn(k * r.n_pix, device="cuda") for k in (3, 1)]
    r.backward(*P, *up, var=True, dL_dmean=up[1], dL_dvar=up[1])
    assert (r.buffer(G.BUF_G2D, torch.float32) != 0).any()
    for which in range(10):
        want = r.buffer(which, torch.uint8)
        odd = torch.zeros(want.numel() + 1, dtype=torch.uint8, device="cuda")
        G.gs_workspace_copy(r.ws, which, ctypes.c_void_p(odd.data_ptr() + 1), want.numel(), G._stream())
        assert torch.equal(odd[1:], want) and odd[0] == 0, which
    r.close()


def test_bytes_a_pair():
    """Record 48, image-space gradient 40, direction gradient 16, rectangle 8,
    depth key 4, the depth sort's double buffers 16, instance offset 4, state 1."""
    from paper_2510_26358_gb300 import gsraster as G
    cam = S.random_box_scene(1, 64, 64, 60.0, seed=0).cameras
    held = []
    for n in (1 << 16, 1 << 20):
        r = G.Renderer(cam, [0, n], 0, inst_capacity=1 << 16)
        held.append(r.info["bytes"])
        r.close()
    assert (held[1] - held[0]) / ((1 << 20) - (1 << 16)) < 138
