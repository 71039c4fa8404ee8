"""The rasterisers divide a tile into 8x8 quadrants and give a warp one, two or
four of them, by the number of tiles; every division must give the same
images bit for bit and the same gradients, and entries whose alpha reaches the
clamp or whose values are not finite must come out as one by one."""
from dataclasses import replace

import numpy as np
import pytest

import oracle as O
from paper_2510_26358_gb300 import scenes as S
from tests.gpu_helpers import rel_l2, run_gpu

pytestmark = pytest.mark.gpu

GRADS = ("g_means", "g_log_scales", "g_quats", "g_opacity_logits", "g_sh")


# 397x401 pixels, 25x26 tiles of 16x16 with a ragged edge of 13 columns and 1
# row: 650 tiles alone, 5200 as 8 views and 41,600 as 64, which lie on either
# side of both lines of the dispatch
@pytest.mark.parametrize("views", [8, 64])
@pytest.mark.parametrize("tile", [(16, 16), (16, 32), (32, 16)])
@pytest.mark.parametrize("var", [False, True])
def test_every_share_renders_alike(views, tile, var):
    sc = S.random_box_scene(1200, 397, 401, 380.0, seed=11, sh_degree=1)
    rng = np.random.default_rng(3)
    n = 397 * 401
    up = [rng.normal(size=k).astype(np.float32) for k in (3 * n, n, n)]
    extra = dict(var=True, gmean=up[1], gvar=0.1 * up[2]) if var else {}
    cfg = O.Config(tile_w=tile[0], tile_h=tile[1])
    one = run_gpu(sc, cfg, *up, **extra)
    many = replace(sc, cameras=sc.cameras * views)
    extra = {k: np.tile(v, views) if k.startswith("g") else v for k, v in extra.items()}
    all_ = run_gpu(many, cfg, *(np.tile(u, views) for u in up), **extra)
    try:
        for k in ("depth", "alpha", "tfin", "last") + (("mean", "var") if var else ()):
            assert np.array_equal(np.tile(one[k].view(np.uint32), views), all_[k].view(np.uint32)), k
        assert np.array_equal(np.tile(one["rgb"].view(np.uint32), views), all_["rgb"].view(np.uint32))
        for k in GRADS:  # sums of the same terms in another order
            assert rel_l2(all_[k], views * one[k].astype(np.float64)) < 1e-5, k
    finally:
        one["renderer"].close()
        all_["renderer"].close()


@pytest.mark.parametrize("views", [1, 64])
def test_clamped_alpha_matches_the_oracle(views):
    """Half of the opacities above alpha_max: their fragments clamp near the
    centre (no gradient through the exponent there)."""
    sc = S.random_box_scene(400, 397, 401, 380.0, seed=12, sh_degree=0, log_scale_mu=-2.5)
    sc.opacity_logits[::2] = 6.0
    P, cams, cfg = O.Params.from_scene(sc), O.as_float32_cameras(sc.cameras), O.Config()
    rec, keys, vals, ranges, out = O.forward(P, cams, cfg)
    ok = out["margin"] > 1e-4
    w = ok.astype(np.float64)
    rng = np.random.default_rng(4)
    up = [(rng.normal(size=k * ok.size) * np.tile(w, k)).astype(np.float32) for k in (3, 1, 1)]
    want = O.render_bwd(P, cams, cfg, rec, vals, ranges, *(u.astype(np.float64) for u in up))
    many = replace(sc, cameras=sc.cameras * views)
    g = run_gpu(many, cfg, *(np.tile(u, views) for u in up))
    try:
        for v in range(views):
            img = g["rgb"].reshape(views, 3, -1)[v].astype(np.float64)
            assert np.abs(img - out["rgb"].reshape(3, -1))[:, ok].max() <= 1e-5
        for k in GRADS:
            assert rel_l2(g[k], views * want[k[2:]]) <= 1e-4, k
    finally:
        g["renderer"].close()


@pytest.mark.parametrize("views", [1, 64])
def test_a_colour_that_is_not_finite_stays_where_it_is_seen(views):
    sc = S.random_box_scene(600, 397, 401, 380.0, seed=13, sh_degree=0)
    # a small Gaussian in front of the others at the image centre
    sc.means[7], sc.log_scales[7], sc.opacity_logits[7] = (0.0, 0.0, 1.5), -5.0, 2.0
    many = replace(sc, cameras=sc.cameras * views)
    a = run_gpu(many, O.Config())
    sc.sh[7, 0, 1] = np.inf
    b = run_gpu(many, O.Config())
    try:
        x, y = (r["rgb"].reshape(views, 3, 401, 397) for r in (a, b))
        assert np.isinf(y[:, 1, 200, 198]).all()
        far = np.ones((401, 397), bool)
        far[185:216, 183:214] = False  # 3.4 sigma of 1.7 pixels, and a margin
        assert np.array_equal(x[:, :, far], y[:, :, far])
        for k in ("depth", "alpha", "tfin", "last"):
            assert np.array_equal(a[k], b[k]), k
    finally:
        a["renderer"].close()
        b["renderer"].close()


# The backward that works entries in pairs stages 32, 64 or 128 of them by the
# number of tiles and the configuration's depth: 397x401 is 2,550 tiles of 8x8 and
# 650 of 16x16, 8 views 20,400 of 8x8; 300x241 is 304 of 16x16.
@pytest.mark.parametrize("size,tile,views", [((397, 401), (8, 8), 1), ((397, 401), (8, 8), 8),
                                             ((397, 401), (16, 16), 1), ((300, 241), (16, 16), 1),
                                             ((300, 241), (16, 32), 1)])
@pytest.mark.parametrize("depth", [32, 128, 256])
@pytest.mark.parametrize("var", [False, True])
def test_backward_in_pairs_gives_the_whole_tiles_gradients(size, tile, views, depth, var):
    sc = S.random_box_scene(5000, *size, 380.0, seed=14, sh_degree=1, log_scale_mu=-2.5)
    sc.opacity_logits[:] -= 3.0  # lists of several hundred entries, blended far down
    rng = np.random.default_rng(5)
    n = size[0] * size[1]
    up = [rng.normal(size=k).astype(np.float32) for k in (3 * n, n, n)]

    def grads(views, cfg, depth):
        extra = dict(var=True, gmean=np.tile(up[1], views), gvar=0.1 * np.tile(up[2], views)) if var else {}
        g = run_gpu(replace(sc, cameras=sc.cameras * views), cfg, *(np.tile(u, views) for u in up), depth=depth,
                    inst_capacity=1 << 24, **extra)
        g["renderer"].close()
        return g

    # 16 views of 16x16 tiles are on the other side of the line: whole tiles a warp
    want = grads(16, O.Config(tile_w=16, tile_h=16), 256)
    got = grads(views, O.Config(tile_w=tile[0], tile_h=tile[1]), depth)
    for k in GRADS:  # either within 1e-5 of 64 bits
        assert rel_l2(got[k].astype(np.float64) / views, want[k].astype(np.float64) / 16) < 2e-5, k
