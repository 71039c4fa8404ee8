"""The binning at the edges of its two dispatch rules: maps up to 16,384 pairs
are compacted, sorted and counted by one block, and tile counts whose bits
9-bit digits sort in fewer passes take those.  Keys, instance order and
ranges must equal the oracle's binning of the same projection bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2510_26358_gb300 import scenes as S
from tests.gpu_helpers import check_binning_stage, run_gpu

pytestmark = pytest.mark.gpu


def _check(sc, tile=(16, 16)):
    cfg = O.Config(tile_w=tile[0], tile_h=tile[1])
    g = run_gpu(sc, cfg)
    try:
        assert g["status"] == 0
        check_binning_stage(sc, cfg, g)
        return g
    finally:
        g["renderer"].close()


@pytest.mark.parametrize("n", [1, 31, 1023, 1025, 2049, 16383, 16384, 16385])
def test_pairs_around_the_one_block_sort(n):
    _check(S.random_box_scene(n, 96, 80, 90.0, seed=n, log_scale_mu=-4.0))


@pytest.mark.parametrize("n", [700, 20_000])
def test_equal_depths_keep_the_pair_order(n):
    """All depths alike, and depths of a handful of values over the whole
    range of floats past the near plane (more than 27 bits apart)."""
    sc = S.random_box_scene(n, 96, 80, 90.0, seed=5, log_scale_mu=-4.0)
    rng = np.random.default_rng(6)
    ratio = sc.means[:, :2] / sc.means[:, 2:]
    for depths in ([3.0], [0.25, 3.0, 3.0000002, 1e5, 3e9]):
        z = rng.choice(np.asarray(depths, np.float32), n)
        sc.means = np.concatenate([ratio * z[:, None], z[:, None]], 1).astype(np.float32)
        sc.log_scales = (-4.0 + np.log(z)[:, None] + np.zeros((n, 3))).astype(np.float32)
        _check(sc)


# 255, 256, 511 and 512 tiles of 16x16 (8, 9, 9 and 10 bits of tile ids and the
# dropped instances' id): one pass of 8 bits, one of 9, two of 8
@pytest.mark.parametrize("size", [(240, 272), (256, 256), (112, 1168), (256, 512)])
@pytest.mark.parametrize("n", [500, 20_000])
def test_tile_counts_around_one_pass(size, n):
    _check(S.random_box_scene(n, *size, 150.0, seed=n + size[0], log_scale_mu=-3.5))


def test_tile_count_of_seventeen_bits():
    """74,240 tiles of 8x8: two passes of 9 bits."""
    sc = S.random_box_scene(20_000, 2560, 1856, 1500.0, seed=9, log_scale_mu=-5.0)
    _check(sc, (8, 8))


def test_capacity_overflow_of_a_small_map():
    """Past the capacity nothing is listed, and the next binning recovers."""
    from paper_2510_26358_gb300 import gsraster as G
    import torch
    from tests.gpu_helpers import params_to_dev
    sc = S.random_box_scene(2000, 96, 80, 90.0, seed=3)
    P = params_to_dev(sc)
    ref = G.Renderer(sc.cameras, sc.submap_offsets, 0, inst_capacity=1 << 20)
    want = ref.forward(*P)
    _, need, _ = ref.status()
    r = G.Renderer(sc.cameras, sc.submap_offsets, 0, inst_capacity=need - 1)
    rgb, _, alpha = r.forward(*P)
    st, n, _ = r.status()
    assert st == G.GS_ERR_CAPACITY and n == need
    assert not rgb.any() and not alpha.any()
    hidden = [*P[:3], torch.full_like(P[3], -9.0), P[4]]  # nothing visible: fits again
    r.forward(*hidden)
    assert r.status()[:2] == (G.GS_OK, 0)
    r.close()
    full = G.Renderer(sc.cameras, sc.submap_offsets, 0, inst_capacity=need)
    assert torch.equal(full.forward(*P)[0], want[0]) and full.status()[0] == G.GS_OK
    full.close()
    ref.close()
