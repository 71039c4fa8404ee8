"""The row copies of the lifecycle, the insertion and the partition at the
edges of their 512-row chunks, for every SH degree (row lengths 3, 12, 27 and
48 words) and for arrays that start on no 16-byte boundary."""
import numpy as np
import pytest

from oracle import lifecycle as L
from oracle import voxel as V
from tests.test_lifecycle_gpu import FIELDS, _compare
from tests.test_lifecycle_oracle import P, random_map

pytestmark = pytest.mark.gpu

SIZES = [1, 511, 512, 513, 1537]


def _array(torch, a, shift):
    """The values of `a` on the GPU, `shift` words past an aligned start."""
    a = np.ascontiguousarray(a)
    buf = torch.zeros(a.size + shift, dtype=torch.from_numpy(a.reshape(-1)).dtype, device="cuda")
    buf[shift:] = torch.from_numpy(a.reshape(-1))
    return buf[shift:].reshape(a.shape)


def _arrays(torch, d, shift):
    return {k: _array(torch, v, shift) for k, v in d.items()}


def _empty(torch, d, rows, shift):
    return _arrays(torch, {k: np.full((rows,) + v.shape[1:], np.nan, np.float32) for k, v in d.items()}, shift)


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("shift", [0, 1])
def test_lifecycle_rows(deg, n, shift):
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    rng = np.random.default_rng(1000 * deg + n)
    offs = (0, n // 3, n // 3, n)
    params, acc, cnt, z, offs = random_map(rng, n, deg=deg, submaps=offs)
    mom = tuple({k: rng.normal(size=v.shape).astype(np.float32) for k, v in params.items()} for _ in range(2))
    ops = L.PRUNE | L.DENSIFY | L.RESET
    out_o, mom_o, offs_o, actions = L.lifecycle(params, mom, offs, acc, cnt, z, P, ops)
    pd, md = _arrays(torch, params, shift), [_arrays(torch, m, shift) for m in mom]
    out, mout = _empty(torch, params, 2 * n, shift), [_empty(torch, params, 2 * n, shift) for _ in range(2)]
    od = torch.as_tensor(offs, dtype=torch.int64, device="cuda")
    offs_g, n_out = torch.empty_like(od), torch.empty(1, dtype=torch.int64, device="cuda")
    stat = [_array(torch, a, 0) for a in (acc, cnt, z)]
    lc, pa, p = G.Lifecycle(n, len(offs) - 1), G.param_arrays, G._ptr
    G.gs_lifecycle_run(lc.lc, G.lifecycle_params(ops, **P), deg, n, len(offs) - 1, p(od), pa(pd), pa(md[0]), pa(md[1]),
                       *map(p, stat), pa(out), pa(mout[0]), pa(mout[1]), 2 * n, p(offs_g), p(n_out), G._stream())
    torch.cuda.synchronize()
    m = int(n_out)
    assert m == out_o["means"].shape[0] and np.array_equal(offs_g.cpu().numpy(), offs_o)
    cut = lambda d: {k: v[:m].cpu().numpy() for k, v in d.items()}
    _compare(params, cut(out), out_o, actions, [cut(x) for x in mout], mom_o)
    for d in (out, *mout):  # nothing past the last row
        for k in FIELDS:
            assert torch.isnan(d[k][m:]).all(), k
    lc.close()


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
def test_partition_rows(deg, n, shift, share):
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    rng = np.random.default_rng(1000 * deg + n)
    params = {k: v.astype(np.float32) for k, v in random_map(rng, n, deg=deg, submaps=(0, n))[0].items()}
    keys, lu = rng.integers(0, 2 ** 62, n), rng.integers(0, 9, n).astype(np.int32)
    f = (rng.random(n) < share).astype(np.int32)
    kept_o, moved_o = V.partition(dict(params, keys=keys, lu=lu), f)
    vm = G.VoxelMap(1, n)
    sides = [(_empty(torch, params, n, shift), torch.zeros(n, dtype=torch.int64, device="cuda"),
              torch.zeros(n, dtype=torch.int32, device="cuda")) for _ in range(2)]
    counts = vm.partition(_array(torch, f, 0), deg, _arrays(torch, params, shift), _array(torch, keys, 0),
                          _array(torch, lu, 0), *sides[0], *sides[1])
    torch.cuda.synchronize()
    assert counts.cpu().tolist() == [n - f.sum(), f.sum()]
    for (arrays, k, u), want in zip(sides, (kept_o, moved_o)):
        m = len(want["keys"])
        for name in params:
            assert np.array_equal(arrays[name][:m].cpu().numpy(), want[name]), name
            assert torch.isnan(arrays[name][m:]).all(), name
        assert np.array_equal(k[:m].cpu().numpy(), want["keys"]) and np.array_equal(u[:m].cpu().numpy(), want["lu"])
    vm.close()


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("n", SIZES)
def test_inserted_rows(deg, n):
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    rng = np.random.default_rng(1000 * deg + n)
    pts = np.concatenate([rng.uniform(-1, 1, (n, 3)), rng.random((n, 3))], 1).astype(np.float32)
    sk, hk = V.keys(pts[::5, :3], 0.1), V.keys(pts[2::7, :3], 0.1)
    lu0 = np.zeros(len(sk), np.int32)
    lu_o, reload_o, new_o, nk_o = V.insert(sk, lu0, hk, pts, 0.1, 9, 0.02, 0.1, deg)
    vm = G.VoxelMap(n, 16)
    lu = _array(torch, lu0, 0)
    reload, new, nk, m = vm.insert(_array(torch, pts, 0), _array(torch, sk.view(np.int64), 0), lu,
                                   _array(torch, hk.view(np.int64), 0), deg, 0.1, 0.02, 0.1, 9)
    assert m == len(nk_o) and np.array_equal(nk.cpu().numpy().view(np.uint64), nk_o)
    assert np.array_equal(lu.cpu().numpy(), lu_o) and np.array_equal(reload.cpu().numpy(), reload_o)
    for k in FIELDS:
        got, want = new[k].cpu().numpy().astype(np.float64), np.asarray(new_o[k]).reshape(new[k].shape)
        assert np.all(np.abs(got - want) <= 1e-6 * (1.0 + np.abs(want))), k
    vm.close()


@pytest.mark.parametrize("n", [2, 255, 256, 257, 4099])
@pytest.mark.parametrize("spread", [1, 3, 1 << 11, 1 << 31])
def test_selection_over_digits(n, spread):
    """Values inside one digit of the radix select, over two of its digits and
    over the whole int32 range, warps that agree on a digit and warps that
    do not."""
    import torch
    from paper_2510_26358_gb300 import gsraster as G
    rng = np.random.default_rng(n)
    lu = rng.integers(-spread, spread, n).astype(np.int32)
    vm = G.VoxelMap(1, n)
    for tau in sorted({0, 1, n // 2, n - 1, n}):
        flags = vm.select(_array(torch, lu, 0), tau)
        assert np.array_equal(flags.cpu().numpy(), V.lru_offload(lu, tau)), tau
    vm.close()
