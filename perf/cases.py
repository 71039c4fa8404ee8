"""The work whose speed this package is judged by, as measurable cases.

A mapping session renders keyframes of a shared Gaussian map from all cameras
of a rig, compares them with the camera images and the LiDAR, back-propagates
to the map and the poses, and now and then updates, prunes, densifies, extends
and pages the map.  Each kind of case below is one of these calls:

  step       one mapping iteration (project, bin, rasterise, losses, backward),
             captured in a CUDA graph once and replayed, as a mapping loop does
  render     a forward pass alone (views of the map for tracking and display)
  pose       forward and backward through torch.autograd (pose refinement)
  image_loss the photometric loss (1 - lambda) L1 + lambda (1 - SSIM) and its gradient
  adam       the optimiser's step over every parameter
  lifecycle  prune, opacity reset, split and clone, with the optimiser's moments
  insert     a keyframe's fused points inserted into the voxel-hashed map
  active     the least recently used splats selected and offloaded to pinned host memory

Scenes are orchard rows (trunks of elongated Gaussians under canopy balls,
seen by rigs of one forward and two lateral cameras) or a random box, made on
the GPU from the seed alone.  ``exact`` evaluates the same formulas densely in
64 bits with plain torch.
"""
from __future__ import annotations

import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2510_26358_gb300 import gsraster as G

PARAMS = G.PARAM_FIELDS
# the renderer's constants as the library holds them (float32)
F32 = lambda x: float(np.float32(x))
NEAR, DILATION, ALPHA_MIN, ALPHA_MAX, T_MIN, CLAMP = map(F32, (0.2, 0.3, 1 / 255, 0.99, 1e-4, 1.3))
SIGMA_L = SIGMA_U = F32(0.05)
Y00 = 0.28209479177387814
ADAM_LR = (1.6e-4, 5e-3, 1e-3, 5e-2, 2.5e-3)
SUBMAP_SIZES = ((640, 480), (1280, 720), (1920, 1080))
MAX_PIX_EXACT = 7_000_000  # beyond this the dense 64-bit evaluation takes too long


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest map and camera (320x240, colour only): a step is a chain of short launches
        dict(name="step_small", kind="step", scene="box", n=10_000, views=1, width=320, height=240, sh=0,
             lidar=0, ssim=0.0, depth_loss="l1", tile=16, batch=256),
        # a keyframe of the three-camera rig on a local map, 8-bit camera images, L1 depth
        dict(name="step_keyframe", kind="step", scene="orchard", n=500_000, views=3, width=1280, height=720, sh=3,
             lidar=20_000, ssim=0.0, depth_loss="l1", tile=16, batch=128),
        # the same with every loss on: SSIM and the LiDAR term with the rendered variance; undistorted
        # (cropped, odd-sized) images, a lower SH degree
        dict(name="step_all_losses", kind="step", scene="orchard", n=300_000, views=3, width=1237, height=701, sh=2,
             lidar=20_000, ssim=0.2, depth_loss="kl-var", tile=16, batch=128),
        # the large keyframe map: two rigs of 1920x1200 over 4M Gaussians, KL depth, dense LiDAR
        dict(name="step_large", kind="step", scene="orchard", n=4_000_000, views=6, width=1920, height=1200, sh=3,
             lidar=100_000, ssim=0.0, depth_loss="kl", tile=16, batch=128),
        # a preview of a small map in one odd-sized view, call by call
        dict(name="render_small", kind="render", scene="box", n=3_001, views=1, width=161, height=119, sh=1,
             var=False, tile=16, batch=256),
        # every camera of eight uneven submaps at once (mixed resolutions), forward only
        dict(name="render_submaps", kind="render", scene="submaps", n=4_400_000, views=24, width=0, height=0, sh=3,
             var=False, tile=16, batch=128),
        # pose refinement of a four-camera rig (perturbed poses) through torch.autograd
        dict(name="pose_rig", kind="pose", scene="orchard", n=1_000_000, views=4, width=1440, height=1080, sh=3,
             tile=16, batch=256),
        # Eq. 6 on a rig's images
        dict(name="image_loss", kind="image_loss", views=3, width=1280, height=720, ssim=0.2),
        # the optimiser after a step on a 1M map
        dict(name="adam", kind="adam", n=1_000_000, sh=3),
        # densification and pruning of a 1M map in four submaps, moments carried along
        dict(name="lifecycle", kind="lifecycle", n=1_000_000, sh=3, submaps=4, moments=True, densify=0.1),
        # a LiDAR keyframe inserted into a 500k map with 100k splats on the host
        dict(name="insert", kind="insert", points=300_000, n=500_000, host=100_000, sh=3),
        # a fifth of a 500k map offloaded to the host store
        dict(name="active_set", kind="active", n=500_000, sh=3, keep=0.8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "render", "render", "pose", "image_loss", "adam", "lifecycle", "insert",
                       "active"])
    sh = rng.choice([0, 1, 2, 3, 3, 3])
    tile, batch = rng.choice([16, 16, 16, 16, 8, 32]), rng.choice([64, 128, 128, 256])
    views = rng.randint(1, 6)
    # image sizes from 160x120 to 1920x1200, odd ones among them
    width = _log_int(rng, 160, 1920)
    height = max(100, min(1200, int(width * rng.uniform(0.55, 0.8))))
    if kind in ("step", "render", "pose"):
        views = max(1, min(views, 8_000_000 // (width * height)))
        box = rng.random() < 0.2
        c = dict(kind=kind, scene="box" if box else "orchard", n=_log_int(rng, 3_000, 60_000 if box else 2_500_000),
                 views=1 if box else views, width=width, height=height, sh=sh)
        if kind == "step":
            c.update(lidar=rng.choice([0, _log_int(rng, 1_000, 100_000)]), ssim=rng.choice([0.0, 0.0, 0.2]),
                     depth_loss=rng.choice(["l1", "kl", "kl-var"]))
        elif kind == "render":
            c.update(var=rng.random() < 0.4)
        c.update(tile=tile, batch=batch)
        return c
    if kind == "image_loss":
        return dict(kind=kind, views=views, width=width, height=height, ssim=rng.choice([0.0, 0.2, 0.5, 1.0]))
    if kind == "adam":
        return dict(kind=kind, n=_log_int(rng, 10_000, 2_000_000), sh=sh)
    if kind == "lifecycle":
        return dict(kind=kind, n=_log_int(rng, 10_000, 2_000_000), sh=sh, submaps=rng.randint(1, 8),
                    moments=rng.random() < 0.7, densify=round(rng.uniform(0.02, 0.3), 3))
    if kind == "insert":
        return dict(kind=kind, points=_log_int(rng, 2_000, 600_000), n=_log_int(rng, 10_000, 2_000_000),
                    host=rng.choice([0, _log_int(rng, 1_000, 300_000)]), sh=sh)
    return dict(kind=kind, n=_log_int(rng, 10_000, 2_000_000), sh=sh, keep=round(rng.uniform(0.5, 0.95), 3))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class _Draws:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)

    def rand(self, *shape):
        return torch.rand(*shape, device="cuda", generator=self.gen)

    def randn(self, *shape):
        return torch.randn(*shape, device="cuda", generator=self.gen)

    def randint(self, lo, hi, n, dtype=torch.int64):
        return torch.randint(lo, hi, (n,), device="cuda", generator=self.gen, dtype=dtype)


def _sh_rows(n, sh, d, rgb=None):
    K = (sh + 1) ** 2
    c = 0.2 * d.randn(n, K, 3)
    if rgb is not None:
        c[:, 0] = (rgb - 0.5) / Y00
    return c


def _box(n, sh, d):
    lo, hi = torch.tensor([-2.0, -1.5, 1.0], device="cuda"), torch.tensor([2.0, 1.5, 7.0], device="cuda")
    return dict(means=lo + (hi - lo) * d.rand(n, 3), log_scales=-3.0 + 0.5 * d.randn(n, 3),
                quats=torch.nn.functional.normalize(d.randn(n, 4), dim=1), opacity_logits=d.randn(n),
                sh=_sh_rows(n, sh, d, d.rand(n, 3)))


def _orchard(n, rows, per_row, sh, d, x0=0.0):
    """Trees 1.5 m apart in rows 3.5 m apart; of a tree's Gaussians one in eleven is trunk."""
    trees = rows * per_row
    # a tree's Gaussians are consecutive, so its neighbours in space are neighbours in memory
    tree = torch.div(torch.arange(n, device="cuda") * trees, n, rounding_mode="floor")
    tx = x0 + 1.5 * (tree % per_row)
    ty = 3.5 * (torch.div(tree, per_row, rounding_mode="floor") - (rows - 1) / 2.0)
    trunk = d.rand(n) < 1.0 / 11.0
    ang, h = 2 * math.pi * d.rand(n), d.rand(n)
    on_trunk = torch.stack([tx + 0.08 * torch.cos(ang), ty + 0.08 * torch.sin(ang), h], 1)
    ball = torch.nn.functional.normalize(d.randn(n, 3), dim=1) * (1.2 * d.rand(n, 1) ** (1 / 3))
    in_canopy = torch.stack([tx, ty, torch.full_like(tx, 2.2)], 1) + ball
    ls_trunk = torch.tensor([-4.5, -4.5, -2.5], device="cuda") + 0.2 * d.randn(n, 3)
    upright = torch.tensor([1.0, 0.0, 0.0, 0.0], device="cuda").expand(n, 4)
    t = trunk[:, None]
    return dict(means=torch.where(t, on_trunk, in_canopy).contiguous(),
                log_scales=torch.where(t, ls_trunk, -4.0 + 0.6 * d.randn(n, 3)).contiguous(),
                quats=torch.where(t, upright, torch.nn.functional.normalize(d.randn(n, 4), dim=1)).contiguous(),
                opacity_logits=d.randn(n), sh=_sh_rows(n, sh, d))


def _camera(center, forward, width, height, submap=0):
    zc = np.asarray(forward, np.float64)
    xc = np.cross(zc, [0.0, 0.0, 1.0])
    R = np.stack([xc, np.cross(zc, xc), zc])
    f = 0.9375 * width
    return SimpleNamespace(width=width, height=height, submap=submap, fx=f, fy=f, cx=width / 2.0, cy=height / 2.0,
                           T_cw=np.concatenate([R, (-R @ np.asarray(center, np.float64))[:, None]], 1))


def _perturbed(cam, rng):
    """Left SE(3) noise of 5 cm and 1 degree."""
    w = np.radians(rng.normal(0.0, 1.0, 3))
    th, K = np.linalg.norm(w), np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
    dR = np.eye(3) + math.sin(th) / th * K + (1 - math.cos(th)) / th ** 2 * (K @ K)
    T = dR @ cam.T_cw
    T[:, 3] += rng.normal(0.0, 0.05, 3)
    return SimpleNamespace(**{**vars(cam), "T_cw": T})


AXES = ((1, 0, 0), (0, 1, 0), (0, -1, 0), (-1, 0, 0))


def _scene(case, seed):
    """(parameters, cameras, submap offsets) of a rendering case."""
    d = _Draws(seed)
    n, sh, W, H = case["n"], case["sh"], case["width"], case["height"]
    if case["scene"] == "box":
        T = np.concatenate([np.eye(3), np.zeros((3, 1))], 1)
        cam = SimpleNamespace(width=W, height=H, submap=0, fx=0.9375 * W, fy=0.9375 * W, cx=W / 2.0, cy=H / 2.0, T_cw=T)
        return _box(n, sh, d), [cam], [0, n]
    if case["scene"] == "submaps":
        # sizes in geometric progression over a factor of 40, three cameras each
        subs = case["views"] // 3
        share = [40.0 ** (s / max(1, subs - 1)) for s in range(subs)]
        offs = [0] + [int(n * sum(share[: s + 1]) / sum(share)) for s in range(subs)]
        parts, cams, x0 = [], [], 0.0
        for s in range(subs):
            cnt = offs[s + 1] - offs[s]
            per_row = max(2, round(cnt / 66_000))
            parts.append(_orchard(cnt, 3, per_row, sh, d, x0))
            W, H = SUBMAP_SIZES[s % 3]
            cams += [_camera((x0 + 0.75 * (per_row - 1), 1.75, 1.2), a, W, H, s) for a in AXES[:3]]
            x0 += 1.5 * per_row + 10.0
        return {k: torch.cat([p[k] for p in parts]) for k in PARAMS}, cams, offs
    rows = 9 if n > 2_000_000 else 3
    per_row = max(2, round(n / (rows * 18_000)))
    P = _orchard(n, rows, per_row, sh, d)
    views = case["views"]
    rig = AXES if views == 4 else AXES[:3]
    cams = []
    for k in range(views):  # one rig a lane, lanes from the middle outwards
        lane = k // len(rig)
        y = 1.75 + 3.5 * ((lane + 1) // 2) * (1 if lane % 2 else -1) if rows > 3 else (1.75 if lane % 2 == 0 else -1.75)
        cams.append(_camera((0.75 * (per_row - 1), y, 1.2), rig[k % len(rig)], W, H))
    if case["kind"] == "pose":
        rng = np.random.Generator(np.random.PCG64(seed))
        cams = [_perturbed(c, rng) for c in cams]
    return P, cams, [0, n]


def _lidar(P, cams, per_view, d):
    """`per_view` returns (u, v, z, view) in every view: map points with 3 cm of range noise, the nearer half of
    those the camera sees, padded with returns outside the image where it sees too few."""
    out = []
    for v, c in enumerate(cams):
        T = torch.tensor(c.T_cw, dtype=torch.float32, device="cuda")
        pick = d.randint(0, P["means"].shape[0], 16 * per_view)
        p = P["means"][pick] @ T[:, :3].T + T[:, 3]
        z = p[:, 2] + 0.03 * d.randn(len(pick))
        u, w = c.fx * p[:, 0] / p[:, 2] + c.cx, c.fy * p[:, 1] / p[:, 2] + c.cy
        ok = (p[:, 2] > 0.3) & (u >= 0) & (u < c.width) & (w >= 0) & (w < c.height)
        order = torch.where(ok, z, torch.full_like(z, 1e9)).argsort(stable=True)[: 2 * per_view: 2]
        row = torch.stack([u, w, z, torch.full_like(z, v)], 1)
        out.append(torch.where(ok[:, None], row, torch.tensor([-1.0, -1.0, 1.0, v], device="cuda"))[order])
    return torch.cat(out).contiguous()


def _images(n_img, width, height, d):
    """Smooth images (coarse random fields) with a little noise, planar, one after another."""
    coarse = d.rand(n_img, 3, max(2, height // 40), max(2, width // 40))
    x = torch.nn.functional.interpolate(coarse, size=(height, width), mode="bilinear", align_corners=True)
    return (x + 0.02 * d.randn(n_img, 3, height, width)).clamp_(0, 1).reshape(-1).contiguous()


def _config(case):
    tw, th = {8: (8, 8), 16: (16, 16), 32: (16, 32)}[case["tile"]]
    mode = 1 if case.get("depth_loss") == "kl" else 0
    return G.gs_config_default(tile_w=tw, tile_h=th, batch_depth=case["batch"], depth_mode=mode)


def _renderer(case, P, cams, offs):
    """A renderer whose instance capacity has been checked on this map, as a program does before its loop."""
    # pairs of the cameras with their own submaps; small maps in large images cover more tiles a pair
    pairs = sum(offs[c.submap + 1] - offs[c.submap] for c in cams)
    per = 64 if case["tile"] == 8 else 16
    cap = max(1 << 20, min(per * pairs, 48 << 20))
    for _ in range(2):
        r = G.Renderer(cams, offs, case["sh"], config=_config(case), inst_capacity=cap)
        r.forward(*(P[k] for k in PARAMS))
        status, need, _visible = r.status()
        if status == G.GS_OK:
            return r
        r.close()
        cap = int(1.1 * need)
    raise RuntimeError("the instance capacity does not suffice")


def _prepare_step(case, seed):
    P, cams, offs = _scene(case, seed)
    d = _Draws(seed + 1_000_003)
    s = SimpleNamespace(case=case, P=[P[k] for k in PARAMS], var=case["depth_loss"] == "kl-var")
    s.r = r = _renderer(case, P, cams, offs)
    e = lambda n: torch.empty(n, device="cuda")
    s.out = [e(3 * r.n_pix)] + [e(r.n_pix) for _ in range(4 if s.var else 2)]
    # camera images: 8-bit for the L1 term, float for SSIM
    s.target = d.rand(3 * r.n_pix)
    if case["ssim"] == 0:
        s.target = (s.target * 256).to(torch.uint8)
    s.lidar = _lidar(P, cams, case["lidar"], d) if case["lidar"] else torch.zeros(0, 4, device="cuda")
    s.loss_rgb, s.loss_depth = torch.zeros(3, device="cuda"), torch.zeros(1, device="cuda")
    s.g_rgb = e(3 * r.n_pix)
    s.g_depth = [e(r.n_pix) for _ in range(2 if s.var else 1)]
    s.grads = {k: torch.empty_like(P[k]) for k in PARAMS}
    s.grads.update(pose=e((r.n_views, 6)), densify_acc=e(r.n),
                   densify_cnt=torch.empty(r.n, dtype=torch.int32, device="cuda"))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        _step(s)
    torch.cuda.current_stream().wait_stream(side)
    s.graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s.graph):
        _step(s)
    s.result = dict(rgb=s.out[0], depth=s.out[1], alpha=s.out[2], loss_depth=s.loss_depth,
                    loss_rgb=s.loss_rgb if case["ssim"] else s.loss_rgb[:1], **s.grads)
    if s.var:
        s.result.update(mean=s.out[3], variance=s.out[4])
    return s


def _step(s):
    r, p, st = s.r, G._ptr, G._stream()
    G.gs_zero_buffers([s.g_rgb, *s.g_depth])
    r.forward(*s.P, outputs=s.out, var=s.var)
    if s.case["ssim"]:
        G.gs_image_loss(r.ws, p(s.out[0]), p(s.target), s.case["ssim"], p(s.loss_rgb), p(s.g_rgb), st)
    else:
        G.gs_image_l1_u8(r.ws, p(s.out[0]), p(s.target), p(s.loss_rgb), p(s.g_rgb), st)
    m = s.lidar.shape[0]
    if s.var:
        G.gs_depth_loss_var(r.ws, p(s.out[2]), p(s.out[3]), p(s.out[4]), p(s.lidar), m, p(s.loss_depth),
                            p(s.g_depth[0]), p(s.g_depth[1]), st)
        r.backward(*s.P, s.g_rgb, None, grads=s.grads, overwrite=True, var=True, dL_dmean=s.g_depth[0],
                   dL_dvar=s.g_depth[1])
    else:
        G.gs_depth_loss(r.ws, p(s.out[1]), p(s.out[2]), p(s.lidar), m, p(s.loss_depth), p(s.g_depth[0]), st)
        r.backward(*s.P, s.g_rgb, s.g_depth[0], grads=s.grads, overwrite=True)


def _prepare_render(case, seed):
    P, cams, offs = _scene(case, seed)
    return SimpleNamespace(case=case, P=[P[k] for k in PARAMS], r=_renderer(case, P, cams, offs))


def _prepare_pose(case, seed):
    P, cams, offs = _scene(case, seed)
    s = SimpleNamespace(case=case, r=_renderer(case, P, cams, offs))
    s.leaves = [P[k].requires_grad_() for k in PARAMS] + [torch.zeros(len(cams), 6, device="cuda", requires_grad=True)]
    d = _Draws(seed + 1_000_003)
    s.up = [d.randn(3 * s.r.n_pix), d.randn(s.r.n_pix), d.randn(s.r.n_pix)]
    s.fn = G.GSRender()
    return s


def _image_inputs(case, seed):
    d = _Draws(seed)
    y = _images(case["views"], case["width"], case["height"], d)
    return (y + 0.05 * d.randn(y.numel())).clamp_(0, 1), y


def _prepare_image_loss(case, seed):
    x, y = _image_inputs(case, seed)
    cams = [_camera((0, 0, 0), AXES[0], case["width"], case["height"]) for _ in range(case["views"])]
    r = G.Renderer(cams, [0, 1], 0, inst_capacity=1 << 20)
    return SimpleNamespace(case=case, r=r, x=x, y=y, g=torch.zeros_like(x))


def _map(n, sh, d):
    return _orchard(n, 3, max(2, round(n / 54_000)), sh, d)


def _adam_inputs(case, seed):
    d = _Draws(seed)
    P = _map(case["n"], case["sh"], d)
    grad = {k: 1e-4 * d.randn(*t.shape) for k, t in P.items()}
    m = {k: 1e-4 * d.randn(*t.shape) for k, t in P.items()}
    v = {k: 1e-8 * (0.05 + d.rand(*t.shape)) for k, t in P.items()}
    return P, grad, m, v


def _prepare_adam(case, seed):
    P, grad, m, v = _adam_inputs(case, seed)
    return SimpleNamespace(case=case, P=P, grad=grad, m=m, v=v)


LIFECYCLE = dict(densify_grad=2.0, split_scale=0.03, clone_scale=0.02, reset_opacity=0.3)


def _lifecycle_inputs(case, seed):
    d = _Draws(seed)
    n = case["n"]
    P = _map(n, case["sh"], d)
    P["opacity_logits"] *= 2.5  # some have faded
    cnt = d.randint(0, 7, n, torch.int32)
    # the mean image-space gradient exceeds the threshold for a share of the splats
    acc = cnt * torch.where(d.rand(n) < case["densify"], 2.0 + d.rand(n), 1.9 * d.rand(n))
    mom = tuple({k: 1e-3 * d.randn(*t.shape) for k, t in P.items()} for _ in range(2)) if case["moments"] else None
    cuts = np.linspace(0, 1, case["submaps"] + 1) ** 1.5
    offs = [int(n * x) for x in cuts]
    return P, acc, cnt, d.randn(n, 2, 3), mom, offs


def _prepare_lifecycle(case, seed):
    P, acc, cnt, normals, mom, offs = _lifecycle_inputs(case, seed)
    offs = torch.tensor(offs, device="cuda")
    rows = lambda: {k: torch.zeros((2 * case["n"],) + tuple(t.shape[1:]), device="cuda") for k, t in P.items()}
    return SimpleNamespace(case=case, P=P, acc=acc, cnt=cnt, normals=normals, mom=mom or (None, None), offs=offs,
                           out=rows(), out_mom=(rows(), rows()) if mom else (None, None),
                           out_offs=torch.zeros_like(offs), n_out=torch.zeros(1, dtype=torch.int64, device="cuda"),
                           lc=G.Lifecycle(case["n"], case["submaps"]),
                           lp=G.lifecycle_params(G.GS_LC_PRUNE | G.GS_LC_DENSIFY | G.GS_LC_RESET, **LIFECYCLE))


VOXEL, S_INIT, O_INIT, FRAME = 0.05, 0.02, 0.1, 31


def _insert_inputs(case, seed):
    d = _Draws(seed)
    n, m, h = case["n"], case["points"], case["host"]
    means = _map(n, 0, d)["means"]
    # a fifth of the points on splats of the map, a tenth on splats paged out, the rest on surfaces a little beyond
    base = means[d.randint(0, n, m)]
    new = d.rand(m, 1) < 0.7
    xyz = torch.where(new, base * torch.tensor([1.0, 1.0, 1.05], device="cuda") + 0.3 * d.randn(m, 3),
                      base + 1e-3 * d.rand(m, 3))
    points = torch.cat([xyz, d.rand(m, 3)], 1).contiguous()
    host = points[d.randint(0, m, h), :3] if h else torch.zeros(0, 3, device="cuda")
    host = host + 2.0 * (d.rand(h, 1) < 0.7)  # most of the host's voxels lie elsewhere
    return points, means, host.contiguous(), d.randint(0, 30, n, torch.int32)


def _prepare_insert(case, seed):
    points, means, host, last_used = _insert_inputs(case, seed)
    vm = G.VoxelMap(case["points"], case["n"])
    keys, hkeys = vm.keys(means, VOXEL), vm.keys(host, VOXEL)
    m, K = case["points"], (case["sh"] + 1) ** 2
    new = {k: torch.zeros(m, *shape, device="cuda") for k, shape in zip(PARAMS, ((3,), (3,), (4,), (), (K, 3)))}
    return SimpleNamespace(case=case, vm=vm, points=points, keys=keys, hkeys=hkeys, last_used=last_used, new=new,
                           new_keys=torch.zeros(m, dtype=torch.int64, device="cuda"),
                           n_new=torch.zeros(1, dtype=torch.int64, device="cuda"),
                           reload=torch.zeros(case["host"], dtype=torch.int32, device="cuda"),
                           ip=G.GsInsertParams(VOXEL, S_INIT, O_INIT, FRAME))


def _active_inputs(case, seed):
    d = _Draws(seed)
    n = case["n"]
    return _map(n, case["sh"], d), d.randint(-(1 << 62), 1 << 62, n), d.randint(0, 30, n, torch.int32)


def _prepare_active(case, seed):
    P, keys, last_used = _active_inputs(case, seed)
    n, tau = case["n"], int(case["keep"] * case["n"])
    host = lambda t, rows: torch.empty((rows,) + tuple(t.shape[1:]), dtype=t.dtype).pin_memory()
    dev = lambda t, rows: torch.empty((rows,) + tuple(t.shape[1:]), dtype=t.dtype, device="cuda")
    s = SimpleNamespace(case=case, P=P, keys=keys, lu=last_used, tau=tau, vm=G.VoxelMap(1, n))
    s.kept, s.moved = {k: dev(t, tau) for k, t in P.items()}, {k: host(t, n - tau) for k, t in P.items()}
    s.kept_keys, s.kept_lu = dev(keys, tau), dev(last_used, tau)
    s.moved_keys, s.moved_lu = host(keys, n - tau), host(last_used, n - tau)
    return s


_PREPARE = dict(step=_prepare_step, render=_prepare_render, pose=_prepare_pose, image_loss=_prepare_image_loss,
                adam=_prepare_adam, lifecycle=_prepare_lifecycle, insert=_prepare_insert, active=_prepare_active)


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "step":
        s.graph.replay()
        return s.result
    if kind == "render":
        out = s.r.forward(*s.P, var=case["var"])
        return dict(zip(("rgb", "depth", "alpha", "mean", "variance"), out))
    if kind == "pose":
        out = s.fn.apply(s.r, *s.leaves)
        grads = torch.autograd.grad(out, s.leaves, s.up)
        return dict(zip(("rgb", "depth", "alpha"), (t.detach() for t in out)), **dict(zip(PARAMS + ("pose",), grads)))
    if kind == "image_loss":
        s.g.zero_()
        return dict(loss=s.r.image_loss(s.x, s.y, case["ssim"], s.g), grad=s.g)
    if kind == "adam":
        G.adam_step(s.P, s.grad, s.m, s.v, case["sh"], 500, ADAM_LR)
        return [s.P, s.m, s.v]
    if kind == "lifecycle":
        pa, p = G.param_arrays, G._ptr
        G.gs_lifecycle_run(s.lc.lc, s.lp, case["sh"], case["n"], case["submaps"], p(s.offs), pa(s.P), *map(pa, s.mom),
                           p(s.acc), p(s.cnt), p(s.normals), pa(s.out), *map(pa, s.out_mom), 2 * case["n"],
                           p(s.out_offs), p(s.n_out), G._stream())
        return [s.out, s.out_offs, s.n_out, *s.out_mom]
    if kind == "insert":
        p, m = G._ptr, case["points"]
        status = G.lib().gs_voxel_insert(s.vm.vx, ctypes.byref(s.ip), p(s.points), m, p(s.keys), p(s.last_used),
                                         case["n"], p(s.hkeys), p(s.reload), case["host"], case["sh"],
                                         ctypes.byref(G.param_arrays(s.new)), p(s.new_keys), m, p(s.n_new),
                                         G._stream())
        if status != G.GS_OK:
            raise G.GsError(status, "gs_voxel_insert")
        return [s.reload, s.new, s.new_keys, s.n_new, s.last_used]
    flags = s.vm.select(s.lu, s.tau)
    counts = s.vm.partition(flags, case["sh"], s.P, s.keys, s.lu, s.kept, s.kept_keys, s.kept_lu, s.moved,
                            s.moved_keys, s.moved_lu)
    return [flags, counts, s.kept, s.kept_keys, s.kept_lu, s.moved, s.moved_keys, s.moved_lu]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _sizes(case):
    if case.get("scene") == "submaps":
        subs = case["views"] // 3
        share = [40.0 ** (s / max(1, subs - 1)) for s in range(subs)]
        pix = 3 * sum(SUBMAP_SIZES[s % 3][0] * SUBMAP_SIZES[s % 3][1] for s in range(subs))
        return 3 * case["n"], pix
    return case["views"] * case["n"], case["views"] * case["width"] * case["height"]


def work(case):
    """Bytes: every input read and every output written once.  Flops of the renderer: about 100 per pair projected
    and, with some 80 list entries walked and 47 blended a pixel (counted on the orchards), 1400 per pixel forward
    and 2600 backward."""
    kind = case["kind"]
    if kind == "image_loss":
        n = 3 * case["views"] * case["width"] * case["height"]
        return {"bytes": 16 * n, "flops": (12 + (380 if case["ssim"] else 0)) * n}
    row = 4 * (11 + 3 * (case["sh"] + 1) ** 2)
    n = case["n"]
    if kind == "adam":
        return {"bytes": 7 * row * n, "flops": 12 * row // 4 * n}
    if kind == "lifecycle":
        return {"bytes": (row * (6 if case["moments"] else 2) + 8) * n, "flops": 20 * n}
    if kind == "insert":
        m, h = case["points"], case["host"]
        return {"bytes": 24 * m + 8 * n + 12 * h + (row + 8) * m // 2, "flops": 12 * m}
    if kind == "active":
        return {"bytes": (2 * (row + 12) + 8) * n, "flops": n}
    pairs, pix = _sizes(case)
    bytes_, flops = row * n + 20 * pix, 100 * pairs + 1400 * pix
    if kind == "render":
        return {"bytes": bytes_ + (8 * pix if case["var"] else 0), "flops": flops}
    bytes_, flops = bytes_ + row * n, flops + 2600 * pix + 300 * pairs
    if kind == "pose":
        return {"bytes": bytes_ + 20 * pix, "flops": flops}
    image = 12 * pix if case["ssim"] else 3 * pix
    return {"bytes": bytes_ + image + 8 * n + 16 * case["lidar"] * case["views"], "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, densely, with plain torch
# ---------------------------------------------------------------------------

def _sh_basis(d, deg):
    x, y, z = d.unbind(1)
    pi = math.pi
    Y = [torch.full_like(x, Y00)]
    if deg >= 1:
        Y += [math.sqrt(3 / (4 * pi)) * t for t in (y, z, x)]
    if deg >= 2:
        a = math.sqrt(15 / (4 * pi))
        Y += [a * x * y, a * y * z, math.sqrt(5 / (16 * pi)) * (2 * z * z - x * x - y * y), a * x * z,
              a / 2 * (x * x - y * y)]
    if deg >= 3:
        a, b, c = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
        Y += [a * y * (3 * x * x - y * y), b * x * y * z, c * y * (4 * z * z - x * x - y * y),
              math.sqrt(7 / (16 * pi)) * z * (2 * z * z - 3 * x * x - 3 * y * y), c * x * (4 * z * z - x * x - y * y),
              b / 2 * z * (x * x - y * y), a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


class _View:
    """One camera's view of the Gaussians `ids` in 64 bits: the projected quantities, on the autograd graph of the
    parameters `P` and the pose twist `xi`, and as plain values `q` ordered by depth."""

    def __init__(self, P, sl, cam, deg):
        g = lambda x: F32(x)
        T = torch.tensor(np.asarray(cam.T_cw, np.float32).astype(np.float64), device="cuda")
        W, H, fx, fy, cx, cy = cam.width, cam.height, g(cam.fx), g(cam.fy), g(cam.cx), g(cam.cy)
        self.W, self.H = W, H
        with torch.no_grad():
            z = P["means"][sl] @ T[2, :3] + T[2, 3]
            self.ids = torch.nonzero(z > NEAR).squeeze(1) + sl.start
        self.xi = torch.zeros(6, dtype=torch.float64, device="cuda", requires_grad=True)
        rho, phi = self.xi[:3], self.xi[3:]
        o = torch.zeros((), dtype=torch.float64, device="cuda")
        hat = torch.stack([torch.stack([o, -phi[2], phi[1]]), torch.stack([phi[2], o, -phi[0]]),
                           torch.stack([-phi[1], phi[0], o])])
        R, t = T[:, :3] + hat @ T[:, :3], T[:, 3] + hat @ T[:, 3] + rho
        mu = P["means"][self.ids]
        p = mu @ R.T + t
        x, y, z = p.unbind(1)
        qw, qx, qy, qz = torch.nn.functional.normalize(P["quats"][self.ids], dim=1).unbind(1)
        Rq = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                          2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                          2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)],
                         1).reshape(-1, 3, 3)
        M = R @ (Rq * P["log_scales"][self.ids].exp()[:, None, :])
        lx, ly = CLAMP * max(cx, W - cx) / fx, CLAMP * max(cy, H - cy) / fy
        tx, ty = (x / z).clamp(-lx, lx) / z, (y / z).clamp(-ly, ly) / z
        r0 = fx * (M[:, 0] / z[:, None] - M[:, 2] * tx[:, None])
        r1 = fy * (M[:, 1] / z[:, None] - M[:, 2] * ty[:, None])
        a, b, c = (r0 * r0).sum(1) + DILATION, (r0 * r1).sum(1), (r1 * r1).sum(1) + DILATION
        det = a * c - b * b
        lno = torch.nn.functional.logsigmoid(P["opacity_logits"][self.ids])
        dirs = torch.nn.functional.normalize(mu + R.T @ t, dim=1)
        rgb = (0.5 + torch.einsum("nk,nkc->nc", _sh_basis(dirs, deg), P["sh"][self.ids])).clamp(min=0)
        self.graph = torch.cat([torch.stack([fx * x / z + cx, fy * y / z + cy, c / det, -b / det, a / det, lno], 1),
                                rgb, z[:, None]], 1)
        with torch.no_grad():
            q = self.graph.detach()
            E = 2 * (lno - math.log(ALPHA_MIN))
            ex, ey = (E.clamp(min=0) * a).sqrt() + 0.1, (E.clamp(min=0) * c).sqrt() + 0.1
            box = torch.stack([q[:, 0] - ex, q[:, 0] + ex, q[:, 1] - ey, q[:, 1] + ey], 1)
            seen = (E > 0) & (box[:, 1] > 0) & (box[:, 0] < W) & (box[:, 3] > 0) & (box[:, 2] < H)
            self.order = torch.nonzero(seen).squeeze(1)
            self.order = self.order[q[self.order, 9].float().argsort(stable=True)]
            self.q, self.box = q[self.order], box[self.order]
        self.grad = torch.zeros_like(self.q)

    def blocks(self, size=64):
        for y0 in range(0, self.H, size):
            row = torch.nonzero((self.box[:, 3] > y0) & (self.box[:, 2] < y0 + size)).squeeze(1)
            for x0 in range(0, self.W, size):
                b = self.box[row]
                yield x0, y0, min(self.W, x0 + size), min(self.H, y0 + size), row[(b[:, 1] > x0) & (b[:, 0] < x0 + size)]

    def blend(self, x0, y0, x1, y1, k):
        """Per (Gaussian, pixel) of a block: weight, unclamped alpha, 1 - alpha, transmittance before, offsets."""
        q = self.q[k]
        ys, xs = torch.meshgrid(torch.arange(y0, y1, device="cuda"), torch.arange(x0, x1, device="cuda"), indexing="ij")
        dx = xs.reshape(1, -1) + 0.5 - q[:, 0:1]
        dy = ys.reshape(1, -1) + 0.5 - q[:, 1:2]
        raw = (q[:, 5:6] - 0.5 * (q[:, 2:3] * dx * dx + 2 * q[:, 3:4] * dx * dy + q[:, 4:5] * dy * dy)).exp()
        al = torch.where(raw >= ALPHA_MIN, raw.clamp(max=ALPHA_MAX), torch.zeros_like(raw))
        after = torch.cumprod(1 - al, 0)
        al = torch.where(after >= T_MIN, al, torch.zeros_like(al))
        before = torch.where(al > 0, after / (1 - al), after)
        return q, al * before, raw, al, before, dx, dy

    def forward(self, out, off, var):
        n = self.W * self.H
        rgb = torch.zeros(3, self.H, self.W, dtype=torch.float64, device="cuda")
        maps = [torch.zeros(self.H, self.W, dtype=torch.float64, device="cuda") for _ in range(4)]
        for x0, y0, x1, y1, k in self.blocks():
            if not len(k):
                continue
            q, w = self.blend(x0, y0, x1, y1, k)[:2]
            sh = (y1 - y0, x1 - x0)
            z, Ws = q[:, 9], w.sum(0)
            D = z @ w
            mean = torch.where(Ws > 0, D / Ws.clamp(min=1e-300), D)
            v = (w * (z[:, None] - mean) ** 2).sum(0) if var else Ws
            v = torch.where(Ws > 0, v / Ws.clamp(min=1e-300), v)
            rgb[:, y0:y1, x0:x1] = (q[:, 6:9].T @ w).reshape(3, *sh)
            for m, value in zip(maps, (D, Ws, mean, v)):
                m[y0:y1, x0:x1] = value.reshape(sh)
        out["rgb"][3 * off: 3 * (off + n)] = rgb.reshape(-1)
        for name, m in zip(("depth", "alpha", "mean", "variance"), maps):
            out[name][off: off + n] = m.reshape(-1)

    def backward(self, up, off):
        """Adds to self.grad the adjoint of `forward` for upstream gradients by output name."""
        n = self.W * self.H
        of = lambda name: up[name][off: off + n].reshape(self.H, self.W) if name in up else None
        g_rgb = up["rgb"][3 * off: 3 * (off + n)].reshape(3, self.H, self.W)
        for x0, y0, x1, y1, k in self.blocks():
            if not len(k):
                continue
            cut = lambda m: m[..., y0:y1, x0:x1].reshape(*m.shape[:-2], -1)
            q, w, raw, al, before, dx, dy = self.blend(x0, y0, x1, y1, k)
            z, gc = q[:, 9:10], cut(g_rgb)
            h = q[:, 6:9] @ gc
            gz = torch.zeros_like(w)
            if of("alpha") is not None:
                h = h + cut(of("alpha"))
            if of("depth") is not None:
                h, gz = h + z * cut(of("depth")), gz + cut(of("depth"))
            if of("mean") is not None:
                Ws = w.sum(0).clamp(min=1e-300)
                mean = (z * w).sum(0) / Ws
                v = (w * (z - mean) ** 2).sum(0) / Ws
                a, b = cut(of("mean")) / Ws, cut(of("variance")) / Ws
                h = h + a * (z - mean) + b * ((z - mean) ** 2 - v)
                gz = gz + a + 2 * b * (z - mean)
            wh = w * h
            rest = wh.sum(0) - wh.cumsum(0)
            gp = (before * h - rest / (1 - al)) * torch.where((al > 0) & (raw <= ALPHA_MAX), raw, torch.zeros_like(raw))
            m1, m2 = (gp * dx).sum(1), (gp * dy).sum(1)
            g = torch.stack([q[:, 2] * m1 + q[:, 3] * m2, q[:, 3] * m1 + q[:, 4] * m2, -0.5 * (gp * dx * dx).sum(1),
                             -(gp * dx * dy).sum(1), -0.5 * (gp * dy * dy).sum(1), gp.sum(1)], 1)
            self.grad[k] += torch.cat([g, w @ gc.T, (w * gz).sum(1, keepdim=True)], 1)


def _exact_scene(case, seed, upstream, var=False):
    """Outputs of a rendering case and, where `upstream` makes gradients of them, those of the parameters."""
    P, cams, offs = _scene(case, seed)
    P = {k: t.double().requires_grad_(upstream is not None) for k, t in P.items()}
    pix = [c.width * c.height for c in cams]
    start = [sum(pix[:v]) for v in range(len(cams))]
    out = {k: torch.zeros((3 if k == "rgb" else 1) * sum(pix), dtype=torch.float64, device="cuda")
           for k in ("rgb", "depth", "alpha", "mean", "variance")}
    subs = [slice(offs[c.submap], offs[c.submap + 1]) for c in cams]
    with torch.set_grad_enabled(False):
        for c, sl, o in zip(cams, subs, start):
            _View(P, sl, c, case["sh"]).forward(out, o, var)
    if not var:
        out = {k: out[k] for k in ("rgb", "depth", "alpha")}
    if upstream is None:
        return out
    up, extra = upstream(out, cams)
    acc = torch.zeros(case["n"], dtype=torch.float64, device="cuda")
    pose = []
    for c, sl, o in zip(cams, subs, start):
        view = _View(P, sl, c, case["sh"])
        with torch.no_grad():
            view.backward(up, o)
            acc.index_add_(0, view.ids[view.order], view.grad[:, :2].norm(dim=1))
        view.graph[view.order].backward(view.grad)
        pose.append(view.xi.grad)
    out.update({k: P[k].grad for k in PARAMS}, pose=torch.stack(pose), densify_acc=acc, **extra)
    return out


def _exact_step(case, seed):
    var = case["depth_loss"] == "kl-var"

    def upstream(out, cams):
        P = _scene(case, seed)[0]
        d = _Draws(seed + 1_000_003)
        target = d.rand(out["rgb"].numel())
        target = target.double() if case["ssim"] else (target * 256).to(torch.uint8).float().div(255).double()
        lidar = _lidar(P, cams, case["lidar"], d).double() if case["lidar"] else torch.zeros(0, 4).double().cuda()
        leaf = {k: t.clone().requires_grad_() for k, t in out.items()}
        image = _photometric(leaf["rgb"], target, case["ssim"], cams)
        pix = torch.tensor([c.width * c.height for c in cams], device="cuda")
        W = torch.tensor([c.width for c in cams], device="cuda")
        H = torch.tensor([c.height for c in cams], device="cuda")
        v = lidar[:, 3].long()
        u, w, z = lidar[:, 0], lidar[:, 1], lidar[:, 2]
        ok = (u >= 0) & (u < W[v]) & (w >= 0) & (w < H[v]) & (z > NEAR)
        at = (pix.cumsum(0) - pix)[v[ok]] + w[ok].floor().long() * W[v[ok]] + u[ok].floor().long()
        z, hit = z[ok], out["alpha"][at] > 0
        at, z = at[hit], z[hit]
        if not len(at):
            depth = 0.0 * leaf["depth"].sum() + (0.0 * (leaf["mean"] + leaf["variance"]).sum() if var else 0.0)
        elif case["depth_loss"] == "l1":
            depth = (leaf["depth"][at] - z).abs().mean()
        else:
            s2 = leaf["variance"][at] + SIGMA_U ** 2 if var else torch.full_like(z, SIGMA_U ** 2)
            e = (leaf["mean"] if var else leaf["depth"])[at] - z
            depth = (0.5 * s2.log() - math.log(SIGMA_L) + (SIGMA_L ** 2 + e * e) / (2 * s2) - 0.5).mean()
        (image[0] + depth).backward()
        names = ("rgb", "mean", "variance") if var else ("rgb", "depth")
        extra = dict(loss_rgb=torch.stack(image).detach() if case["ssim"] else image[0].detach().reshape(1),
                     loss_depth=depth.detach().reshape(1))
        return {k: leaf[k].grad for k in names}, extra

    out = _exact_scene(case, seed, upstream, var)
    return dict(out, densify_cnt=None)


def _photometric(x, y, lam, cams):
    """[total, L1, 1 - SSIM] of planar images (only the L1 term when lam is 0)."""
    l1 = (x - y).abs().mean()
    if lam == 0:
        return [l1]
    g = torch.exp(-torch.arange(-5, 6, dtype=torch.float64, device="cuda") ** 2 / 4.5)
    g = g / g.sum()
    blur = lambda t: torch.nn.functional.conv2d(torch.nn.functional.conv2d(t, g.reshape(1, 1, 11, 1), padding=(5, 0)),
                                                g.reshape(1, 1, 1, 11), padding=(0, 5))
    total, o = 0.0, 0
    for c in cams:
        n = 3 * c.width * c.height
        a, b = x[o: o + n].reshape(3, 1, c.height, c.width), y[o: o + n].reshape(3, 1, c.height, c.width)
        o += n
        ma, mb = blur(a), blur(b)
        saa, sbb, sab = blur(a * a) - ma * ma, blur(b * b) - mb * mb, blur(a * b) - ma * mb
        s = (2 * ma * mb + 1e-4) * (2 * sab + 9e-4) / ((ma * ma + mb * mb + 1e-4) * (saa + sbb + 9e-4))
        total = total + (1 - s).sum()
    dssim = total / x.numel()
    return [(1 - lam) * l1 + lam * dssim, l1, dssim]


def _exact_pose(case, seed):
    def upstream(out, _cams):
        d = _Draws(seed + 1_000_003)
        n = out["depth"].numel()
        return dict(zip(("rgb", "depth", "alpha"), (d.randn(k).double() for k in (3 * n, n, n)))), {}

    out = _exact_scene(case, seed, upstream)
    out.pop("densify_acc")
    return out


def _exact_image_loss(case, seed):
    x, y = _image_inputs(case, seed)
    x, y = x.double().requires_grad_(), y.double()
    cams = [SimpleNamespace(width=case["width"], height=case["height"])] * case["views"]
    loss = _photometric(x, y, case["ssim"], cams)
    if case["ssim"] == 0:
        with torch.no_grad():
            loss += [loss[0].detach(), _photometric(x.detach(), y, 0.5, cams)[2]]
    (grad,) = torch.autograd.grad(loss[0], x)
    return dict(loss=torch.stack([t.detach() for t in loss]), grad=grad)


def _exact_adam(case, seed):
    P, grad, m, v = ({k: t.double() for k, t in x.items()} for x in _adam_inputs(case, seed))
    b1, b2 = F32(0.9), F32(0.999)
    for k, lr in zip(PARAMS, ADAM_LR):
        m[k] = b1 * m[k] + (1 - b1) * grad[k]
        v[k] = b2 * v[k] + (1 - b2) * grad[k] ** 2
        P[k] = P[k] - F32(lr) * (m[k] / (1 - b1 ** 500)) / ((v[k] / (1 - b2 ** 500)).sqrt() + F32(1e-15))
    return [P, m, v]


def _exact_lifecycle(case, seed):
    P, acc, cnt, normals, mom, offs = _lifecycle_inputs(case, seed)
    lp = G.lifecycle_params(0, **LIFECYCLE)
    logit = lambda o: F32(math.log(o / (1 - o)))
    ln = lambda s: F32(math.log(s))
    om, s = P["opacity_logits"], P["log_scales"].max(1).values
    lo = logit(lp.prune_opacity)
    gone = (om < lo) | (s > ln(lp.prune_scale_max)) | (s < ln(lp.prune_scale_min))
    reset = (om > lo) & (om < logit(lp.reset_opacity)) & (s > ln(lp.reset_scale_min)) & (s < ln(lp.reset_scale_max))
    dense = torch.where(cnt > 0, acc / cnt, torch.zeros_like(acc)) > lp.densify_grad
    split = dense & (s > ln(lp.split_scale))
    clone = dense & ~split & (s <= ln(lp.clone_scale))
    count = torch.where(gone, 0, torch.where(split | clone, 2, 1))
    src = torch.repeat_interleave(torch.arange(case["n"], device="cuda"), count)
    first = count.cumsum(0) - count
    k = torch.arange(len(src), device="cuda") - first[src]
    out = {name: t.double()[src] for name, t in P.items()}
    out["opacity_logits"] = torch.where(reset[src], logit(lp.reset_opacity), out["opacity_logits"])
    qw, qx, qy, qz = torch.nn.functional.normalize(out["quats"], dim=1).unbind(1)
    R = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                     2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                     2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)], 1).reshape(-1, 3, 3)
    step = (R @ (out["log_scales"].exp() * normals.double()[src, k])[:, :, None]).squeeze(2)
    child = split[src][:, None]
    out["means"] = torch.where(child, out["means"] + step, out["means"])
    out["log_scales"] = torch.where(child, out["log_scales"] - math.log(lp.split_shrink), out["log_scales"])
    rows = lambda x: {name: torch.cat([t, t.new_zeros(2 * case["n"] - len(src), *t.shape[1:])]) for name, t in x.items()}
    result = [rows(out), None, None]
    fresh = split[src] | (clone[src] & (k == 1))
    for m in mom or (None, None):
        result.append(m and rows({name: torch.where(fresh.reshape(-1, *[1] * (t.dim() - 1)), 0.0, t.double()[src])
                                  for name, t in m.items()}))
    return result


def _exact_insert(case, seed):
    points, means, host, _last = _insert_inputs(case, seed)
    primes = torch.tensor([73856093, 19349663, 83492791], device="cuda")
    v = torch.tensor(VOXEL, dtype=torch.float32, device="cuda")
    key = lambda x: (torch.floor(x[:, :3] / v).long() * primes).sum(1)
    pk = key(points)
    uniq, inverse = torch.unique(pk, return_inverse=True)
    first = torch.full((len(uniq),), len(pk), device="cuda").scatter_reduce(
        0, inverse, torch.arange(len(pk), device="cuda"), "amin")
    known = torch.isin(uniq, key(means)) | (torch.isin(uniq, key(host)) if len(host) else False)
    at = first[~known].sort().values
    n, K = len(at), (case["sh"] + 1) ** 2
    full = lambda *shape, value: torch.full(shape, value, dtype=torch.float64, device="cuda")
    sh = full(n, K, 3, value=0.0)
    sh[:, 0] = (points[at, 3:].double() - 0.5) / Y00
    quats = full(n, 4, value=0.0)
    quats[:, 0] = 1.0
    s_init, o_init = F32(S_INIT), F32(O_INIT)
    new = dict(means=points[at, :3].double(), log_scales=full(n, 3, value=math.log(s_init)), quats=quats,
               opacity_logits=full(n, value=math.log(o_init / (1 - o_init))), sh=sh)
    rest = len(points) - n
    new = {k: torch.cat([t, t.new_zeros(rest, *t.shape[1:])]) for k, t in new.items()}
    return [None, new, None, None, None]


def _exact_active(case, seed):
    P, _keys, lu = _active_inputs(case, seed)
    tau = int(case["keep"] * case["n"])
    order = lu.argsort(stable=True)
    flag = torch.zeros(case["n"], dtype=torch.bool, device="cuda")
    flag[order[: case["n"] - tau]] = True
    part = lambda f: {k: t[f].double() for k, t in P.items()}
    return [None, None, part(~flag), None, None, part(flag), None, None]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "render", "pose"):
        if _sizes(case)[1] > MAX_PIX_EXACT or case["n"] > 1_500_000:
            return None
        if kind == "render":
            return _exact_scene(case, seed, None, case["var"])
        return _exact_step(case, seed) if kind == "step" else _exact_pose(case, seed)
    return dict(image_loss=_exact_image_loss, adam=_exact_adam, lifecycle=_exact_lifecycle, insert=_exact_insert,
                active=_exact_active)[kind](case, seed)
