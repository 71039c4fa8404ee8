"""The gradients of large renders are sums whose terms and order are fixed: a
long thin Gaussian near a camera adds thousands of tile sums that largely
cancel, so another order of the same terms moves its gradients past what a
caller may expect of the same inputs.  Here each Gaussian lies inside one tile,
which makes its image-space row one tile's sum, the same bits in every run; the
rows' checksums were recorded from the column-wise sums."""
import zlib

import numpy as np
import pytest

import oracle as O
from paper_2510_26358_gb300 import scenes as S
from tests.gpu_helpers import run_gpu

pytestmark = pytest.mark.gpu

# 4096 tiles of 16x16 (as many pixels of the other sizes), a Gaussian in the middle of every 32x32 pixels' first 8x8
SIZE, PITCH, Z = 1024, 32, 4.0

# (32x16 tiles with the variance split the 8x8 between two warps, which add in either order)
RECORDED = {((8, 8), False): 0x2ffad1b6, ((16, 16), False): 0x6e25aea6, ((16, 32), False): 0x6e25aea6,
            ((32, 16), False): 0x6e25aea6, ((8, 8), True): 0x268f9c6e, ((16, 16), True): 0x0d72e854,
            ((16, 32), True): 0x0d72e854}


def _rows(tile, var, size=SIZE):
    sc = S.random_box_scene((size // PITCH) ** 2, size, size, 960.0, seed=21, sh_degree=0)
    rng = np.random.default_rng(22)
    n = len(sc.means)
    j, i = np.divmod(np.arange(n), size // PITCH)
    at = np.stack([PITCH * i, PITCH * j], 1) + 4.0 + rng.uniform(-0.6, 0.6, (n, 2))
    cam = sc.cameras[0]
    sc.means[:, :2] = (at - [cam.cx, cam.cy]) / [cam.fx, cam.fy] * Z
    sc.means[:, 2] = Z
    sc.log_scales[:] = -8.0
    sc.log_scales[np.arange(n), rng.integers(0, 3, n)] = -5.9  # 0.66 pixels long: 3 sigma stay inside the 8x8
    up = [rng.normal(size=k * size * size).astype(np.float32) for k in (3, 1, 1)]
    extra = dict(var=True, gmean=up[1], gvar=up[2]) if var else {}
    g = run_gpu(sc, O.Config(tile_w=tile[0], tile_h=tile[1]), *up, **extra)
    g["renderer"].close()
    assert (g["pkey"] != 0xFFFFFFFF).all() and len(g["inst_pair"]) == n  # all seen, each in one tile
    return g["g2d"]


@pytest.mark.parametrize("tile,var", RECORDED)
def test_a_tile_sums_its_columns(tile, var):
    rows = _rows(tile, var)
    assert rows.all(1).any() and np.isfinite(rows).all()
    assert zlib.crc32((rows + 0.0).tobytes()) == RECORDED[tile, var]


@pytest.mark.parametrize("var,recorded", [(False, 0xae5396aa), (True, 0x029aee3a)])
def test_tiles_of_8x8_take_columns_sooner(var, recorded):
    # 10,000 tiles: in pairs of entries they took 8 to 15 % longer
    assert zlib.crc32((_rows((8, 8), var, 800) + 0.0).tobytes()) == recorded
