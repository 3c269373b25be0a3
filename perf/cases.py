"""The work that programs have this framework do, as measurable cases.

``listed()`` names twelve cases over the public entry points: training steps of
one view (``pipeline.Trainer``) and of several (``batched.MultiViewTrainer``),
the differentiable renderer (``autograd.render_sampled``), the dense refresh of
an error map, the tile-error network, and the view draw.  ``draw(rng)`` gives
more cases of the same ranges.  ``prepare`` makes what a program holds before
the call, ``run`` is one pass, ``work`` what a pass cannot do without, and
``exact`` the same outputs in 64-bit torch arithmetic.

Training cases stand for a run in its late phase: the optimiser's moments are
filled and the learning rates have decayed to a hundredth of the configured
ones, as position rates do at the end of a 3DGS run.  A scene then keeps its
shape over the thousands of passes that a measurement makes.
"""
import math

import numpy as np
import torch

from paper_2606_15924_gb300 import binding as B
from paper_2606_15924_gb300 import scenes
from paper_2606_15924_gb300.autograd import SampledRaster, render_sampled
from paper_2606_15924_gb300.batched import MultiViewTrainer
from paper_2606_15924_gb300.config import Config, LossConfig, OptConfig
from paper_2606_15924_gb300.pipeline import Trainer, as_geo_rows
from paper_2606_15924_gb300.predictor import TileErrorMLP
from paper_2606_15924_gb300.views import ViewSampler

FIELDS = ("means", "log_scales", "quats", "opacity_logits", "sh")
LR_LATE = 0.01     # learning rates of the late phase, of the configured ones
STEP_LATE = 1000   # the optimiser step that the filled moments stand for


def listed():
    step = dict(kind="step", n=500_000, width=1280, height=720, tiles=0.2, rate=1 / 3, dense=False, rows=True,
                overlap=True, mode=1, structure="ncc", stats=False, sh_degree=3)
    return [
        # the smallest training step: a preview or a unit of a test suite, bound by latency and launches
        dict(step, name="step_tiny_10k", n=10_000, width=256, height=256, tiles=0.25, rows=False, overlap=False),
        # the ordinary sparse step of a scene of half a million Gaussians, as the benchmark runs it
        dict(step, name="step_sparse_500k"),
        # the paper's own sampling: every tile, a tenth of the pixels
        dict(step, name="step_every_tile_500k", tiles=1.0, rate=0.1),
        # the plain dense step (every tile and pixel), the baseline that users compare with
        dict(step, name="step_dense_500k", tiles=1.0, rate=1.0, dense=True),
        # the other options together, at odd sizes: packed arrays, Adam, the S-SSIM loss, density statistics
        dict(step, name="step_options_123k", n=123_457, width=1237, height=821, tiles=0.35, rate=0.25, rows=False,
             overlap=False, mode=0, structure="ssim", stats=True, sh_degree=2),
        # several large views per iteration in one captured step, with uneven tile fractions
        dict(kind="views", name="views_8x3m", n=3_000_000, width=1920, height=1080, views=8, lo=0.03, hi=0.6,
             rate=1 / 3, mode=1),
        # the differentiable renderer inside another program's loop: a small crop ...
        dict(kind="autograd", name="autograd_2k", n=2_000, width=250, height=187, tiles=0.1, sh_degree=3),
        # ... and a large scene
        dict(kind="autograd", name="autograd_2m", n=2_000_000, width=1600, height=1060, tiles=0.2, sh_degree=3),
        # a dense evaluation of one view: its image and its error map, as at set-up and at every plain refresh
        dict(kind="refresh", name="refresh_1m", n=1_000_000, width=1957, height=1091, sh_degree=3),
        # the tile-error network predicts one view's tiles (123 x 69 of them)
        dict(kind="predict", name="predict_view", rows=8_487),
        # and trains on the tiles of a 200-view orbit
        dict(kind="train", name="train_200_views", rows=1_697_400),
        # the view draw over a full view pool
        dict(kind="view_draw", name="view_draw_256", views=256, width=1280, height=720, k=10),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi):
    w = int(_log_uniform(rng, lo, hi))
    return w, max(48, int(w * rng.uniform(0.5, 1.0)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "views", "autograd", "autograd", "refresh", "predict", "train",
                       "view_draw"])
    if kind == "step":
        w, h = _size(rng, 200, 1957)
        dense = rng.random() < 0.25
        every = rng.random() < 0.4
        return dict(kind=kind, n=int(_log_uniform(rng, 5_000, 1_000_000)), width=w, height=h,
                    tiles=1.0 if dense or every else rng.uniform(0.05, 0.6),
                    rate=1.0 if dense else rng.uniform(0.03, 0.34), dense=dense, rows=rng.random() < 0.5,
                    overlap=rng.random() < 0.5, mode=rng.choice([0, 1]), structure=rng.choice(["ncc", "ncc", "ssim"]),
                    stats=rng.random() < 0.25, sh_degree=rng.choice([0, 1, 2, 3, 3, 3]))
    if kind == "views":
        w, h = _size(rng, 300, 1280)
        return dict(kind=kind, n=int(_log_uniform(rng, 20_000, 1_000_000)), width=w, height=h,
                    views=rng.randint(2, 6), lo=0.03, hi=0.6, rate=rng.uniform(0.1, 0.34), mode=rng.choice([0, 1, 2]))
    if kind == "autograd":
        w, h = _size(rng, 100, 1600)
        return dict(kind=kind, n=int(_log_uniform(rng, 1_000, 2_000_000)), width=w, height=h,
                    tiles=rng.uniform(0.03, 0.3), sh_degree=rng.choice([0, 1, 2, 3, 3, 3]))
    if kind == "refresh":
        w, h = _size(rng, 200, 1957)
        return dict(kind=kind, n=int(_log_uniform(rng, 5_000, 1_000_000)), width=w, height=h,
                    sh_degree=rng.choice([0, 1, 2, 3, 3, 3]))
    if kind in ("predict", "train"):
        return dict(kind=kind, rows=int(_log_uniform(rng, 64, 1_700_000)))
    w, h = _size(rng, 100, 1280)
    v = int(_log_uniform(rng, 8, 256))
    return dict(kind=kind, views=v, width=w, height=h, k=rng.randint(3, min(16, v)))


# ---------------------------------------------------------------------------
# inputs, on the GPU, from the seed alone
# ---------------------------------------------------------------------------

def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + what)
    return g


def _extent(n):
    """Half side of the cube of means and the camera's distance: a small object, or a scene."""
    return (1.0, 4.0) if n < 50_000 else (5.0, 15.0)


def _scene(n, seed):
    """n Gaussians of the synthetic scenes' distributions (scenes.gaussians), drawn on the GPU."""
    g, e = _gen(seed, 1), _extent(n)[0]

    def normal(*s):
        return torch.randn(*s, device="cuda", generator=g)
    q = normal(n, 4)
    return dict(means=(torch.rand(n, 3, device="cuda", generator=g) * 2 - 1) * e, log_scales=normal(n, 3) * 0.5 - 3.5,
                quats=q / q.norm(dim=1, keepdim=True), opacity_logits=normal(n), sh=normal(n, 16, 3) * 0.2)


def _camera(n, width, height, azimuth=0.0):
    d, el = _extent(n)[1], math.radians(20.0 if azimuth else 0.0)
    pos = (d * math.cos(el) * math.sin(azimuth), -d * math.sin(el), -d * math.cos(el) * math.cos(azimuth))
    return scenes.look_at(pos, width=width, height=height)


def _image(width, height, seed, what):
    """A smooth colour image in [0, 1] with pixel noise of 0.01."""
    g = _gen(seed, what)
    low = torch.rand(1, 3, 8, 12, device="cuda", generator=g)
    img = torch.nn.functional.interpolate(low, size=(height, width), mode="bicubic", align_corners=False)
    img = img + 0.01 * torch.randn(img.shape, device="cuda", generator=g)
    return img[0].permute(1, 2, 0).clamp(0.0, 1.0).contiguous()


def _error_map(width, height, seed, what):
    """fp16 error map of a partly fitted view: a half-normal background and hot regions (as int16 bits)."""
    g = _gen(seed, what)
    low = torch.rand(1, 1, 9, 16, device="cuda", generator=g) ** 4
    hot = torch.nn.functional.interpolate(low, size=(height, width), mode="bilinear", align_corners=False)[0, 0]
    e = 0.1 * torch.randn(height, width, device="cuda", generator=g).abs() + 0.8 * hot
    return e.half().view(torch.int16)


def _age_map(width, height, seed, what):
    return torch.randint(0, 201, (height, width), device="cuda", generator=_gen(seed, what), dtype=torch.int16)


def _moments(params, seed):
    """First and second moments of an optimiser that has run for a while."""
    g = _gen(seed, 5)
    m, v = {}, {}
    for k in FIELDS:
        s = 1e-5 * torch.exp(torch.randn(params[k].shape, device="cuda", generator=g))
        m[k] = 0.3 * s * torch.randn(params[k].shape, device="cuda", generator=g)
        v[k] = s * s
    return m, v


def _config(case):
    o = OptConfig(mode=case["mode"])
    for k in ("lr_means", "lr_scales", "lr_quats", "lr_opacity", "lr_sh_dc", "lr_sh_rest"):
        setattr(o, k, getattr(o, k) * LR_LATE)
    return Config(opt=o, loss=LossConfig(structure=case.get("structure", "ncc")))


def _into(dst, src):
    for k in FIELDS:
        dst[k].copy_(src[k])


def _late_phase(tr, scene, seed):
    """The captured trainer's state back to the scene, with filled moments (capturing ran one step)."""
    m, v = _moments(scene, seed)
    _into(tr.params, scene)
    _into(tr.m, m)
    _into(tr.v, v)
    tr.step_dev.fill_(STEP_LATE)


def _prepare_step(case, seed):
    scene = _scene(case["n"], seed)
    params = as_geo_rows(scene) if case["rows"] else {k: v.clone() for k, v in scene.items()}
    W, H = case["width"], case["height"]
    tr = Trainer(params, _camera(case["n"], W, H), _image(W, H, seed, 2), tile_fraction=case["tiles"],
                 pixel_rate=case["rate"], cfg=_config(case), dense=case["dense"], seed=int(seed) & 0xFFFF,
                 sh_degree=case["sh_degree"], stats=case["stats"])
    tr.err_map.copy_(_error_map(W, H, seed, 3))
    tr.age_map.copy_(_age_map(W, H, seed, 4))
    tr.capture(overlap=case["overlap"])
    _late_phase(tr, scene, seed)
    tr.err_map.copy_(_error_map(W, H, seed, 3))
    tr.age_map.copy_(_age_map(W, H, seed, 4))
    tr.reset_stats()
    return tr


def _prepare_views(case, seed):
    scene = _scene(case["n"], seed)
    W, H, V = case["width"], case["height"], case["views"]
    fr = np.random.RandomState(int(seed) % (1 << 31)).uniform(case["lo"], case["hi"], V).tolist()
    mv = MultiViewTrainer(as_geo_rows(scene), [_camera(case["n"], W, H, 2 * math.pi * (k + 0.5) / V) for k in range(V)],
                          [_image(W, H, seed, 10 + k) for k in range(V)], fr, pixel_rate=case["rate"],
                          cfg=_config(case), seed=int(seed) & 0xFFFF)
    for k, v in enumerate(mv.views):
        v.err_map.copy_(_error_map(W, H, seed, 30 + k))
        v.age_map.copy_(_age_map(W, H, seed, 50 + k))
    mv.capture()
    _late_phase(mv, scene, seed)
    for k, v in enumerate(mv.views):
        v.err_map.copy_(_error_map(W, H, seed, 30 + k))
        v.age_map.copy_(_age_map(W, H, seed, 50 + k))
    return mv


def _tile_set(case):
    """The tiles that an autograd case renders: a random set of the given share (one for all seeds, since tiles at
    the image's edge have fewer pixels)."""
    T = ((case["width"] + 15) // 16) * ((case["height"] + 15) // 16)
    k = max(1, round(case["tiles"] * T))
    return sorted(np.random.RandomState(7).choice(T, size=k, replace=False).tolist())


def _tile_pixels(tile, width, height, device="cuda"):
    """x and y of a tile's pixels in the image, row by row."""
    tx_n = (width + 15) // 16
    x0, y0 = 16 * (tile % tx_n), 16 * (tile // tx_n)
    y, x = torch.meshgrid(torch.arange(y0, min(y0 + 16, height), device=device),
                          torch.arange(x0, min(x0 + 16, width), device=device), indexing="ij")
    return x.reshape(-1), y.reshape(-1)


def _prepare_autograd(case, seed):
    W, H = case["width"], case["height"]
    leaves = {k: v.requires_grad_(True) for k, v in _scene(case["n"], seed).items()}
    raster = SampledRaster.from_tiles(_camera(case["n"], W, H), case["n"], _tile_set(case),
                                      sh_degree=case["sh_degree"])
    xy = raster.pixel_coords()
    return dict(params=leaves, raster=raster, target=_image(W, H, seed, 2)[xy[:, 1], xy[:, 0]])


def _prepare_refresh(case, seed):
    W, H = case["width"], case["height"]
    tr = Trainer(_scene(case["n"], seed), _camera(case["n"], W, H), _image(W, H, seed, 2), train=False,
                 sh_degree=case["sh_degree"])
    tr.init_error_map(want_loss=False)  # a program has evaluated its views once at set-up
    return tr


def _features(rows, seed):
    """Tile features of the ranges that the path sees (see tgs_tile_features)."""
    g = _gen(seed, 7)
    u = torch.rand(rows, 7, device="cuda", generator=g)
    x = torch.zeros(rows, 16, device="cuda")
    x[:, 0] = torch.log1p(2000.0 * u[:, 0])
    x[:, 1] = u[:, 1]
    x[:, 2] = torch.log1p(0.5 * u[:, 2])
    x[:, 3] = 2.0 * u[:, 3] - 1.0
    x[:, 4] = torch.log1p(200.0 * u[:, 4])
    x[:, 5] = 0.8 + 0.2 * u[:, 5]
    x[:, 6] = (u[:, 6] < 0.95).float()
    return x


def _prepare_mlp(case, seed):
    x = _features(case["rows"], seed)
    g = _gen(seed, 8)
    target = (0.8 * x[:, 2] + 0.05 * x[:, 4] + 0.02 * torch.randn(case["rows"], device="cuda", generator=g)).contiguous()
    mlp = TileErrorMLP(seed=int(seed) & 0xFFFF, lr=1e-5)
    n = mlp.params.numel()
    s = 1e-3 * torch.exp(torch.randn(n, device="cuda", generator=g))
    mlp.m.copy_(0.3 * s * torch.randn(n, device="cuda", generator=g))
    mlp.v.copy_(s * s)
    mlp.step_count = STEP_LATE
    return dict(mlp=mlp, x=x, target=target)


def _prepare_view_draw(case, seed):
    W, H, V = case["width"], case["height"], case["views"]
    g = _gen(seed, 9)
    maps = torch.empty(V, H, W, dtype=torch.int16, device="cuda")
    for v in range(V):
        level = 0.02 + 0.2 * torch.rand(1, device="cuda", generator=g)
        maps[v] = (torch.rand(H, W, device="cuda", generator=g) * level).half().view(torch.int16)
    cams = scenes.orbit(V, distance=15.0, width=W, height=H, seed=int(seed) & 0xFFFF)
    return dict(sampler=ViewSampler(cams, seed=int(seed) & 0xFFFF), maps=maps, it=0, k=case["k"])


def prepare(case, seed):
    make = dict(step=_prepare_step, views=_prepare_views, autograd=_prepare_autograd, refresh=_prepare_refresh,
                predict=_prepare_mlp, train=_prepare_mlp, view_draw=_prepare_view_draw)[case["kind"]]
    return dict(case=case, held=make(case, seed))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    kind, s = state["case"]["kind"], state["held"]
    if kind in ("step", "views"):
        # the updated parameters and moments; the moments carry the gradient
        s.replay()
        out = dict(params=s.params, m=s.m, v=s.v)
        if kind == "step" and s.stats is not None:
            out.update(stats=s.stats, screen=s.accum)
        return out
    if kind == "autograd":
        rgb = render_sampled(s["params"], s["raster"])
        loss = torch.nn.functional.mse_loss(rgb, s["target"])
        grads = torch.autograd.grad(loss, [s["params"][k] for k in FIELDS])
        return dict(rgb=rgb, grads=dict(zip(FIELDS, grads)))
    if kind == "refresh":
        seen = {}
        s.init_error_map(on_dense=lambda d: seen.update(rgb=d.rgb[:s.W * s.H]), want_loss=False)
        return dict(rgb=seen["rgb"], error=s.err_map.view(torch.float16))
    if kind == "predict":
        return dict(y=s["mlp"].predict(s["x"]))
    if kind == "train":
        s["mlp"].train_step(s["x"], s["target"])
        return dict(grads=s["mlp"].grads, params=s["mlp"].params, m=s["mlp"].m, v=s["mlp"].v)
    s["it"] += 1
    sums = s["sampler"].error_sums(s["maps"])
    return dict(sums=sums, views=s["sampler"].draw(s["k"], s["it"]))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _walk(case):
    """Expected splats in a tile's list, and those that a pixel composites before it saturates."""
    e, d = _extent(case["n"])
    scale = case["width"] / (2.0 * math.tan(math.radians(30.0))) / d   # pixels per unit at the centre
    r = 3.0 * math.sqrt((0.04 * scale) ** 2 + 0.3) + 0.5
    ext = [min(s, 2.0 * e * scale) for s in (case["width"], case["height"])]
    seen = min(1.0, case["width"] / (2.0 * e * scale)) * min(1.0, case["height"] / (2.0 * e * scale))
    pairs = case["n"] * seen * (2.0 * r + 16.0) ** 2 / (ext[0] * ext[1])
    return seen, pairs, min(pairs, 400.0)


def work(case):
    kind = case["kind"]
    if kind in ("predict", "train"):
        # 64 B of features a row, and its output or target; the weights are small
        per = 2.0 * (16 * 128 + 128 * 128 + 128)
        return dict(bytes=68.0 * case["rows"], flops=per * case["rows"] * (3.0 if kind == "train" else 1.0))
    if kind == "view_draw":
        return dict(bytes=2.0 * case["views"] * case["width"] * case["height"], flops=0.0)
    n, pix = case["n"], case["width"] * case["height"]
    seen, pairs, walk = _walk(case)
    if kind == "refresh":
        # 44 B of geometry of every Gaussian, the SH row of the visible ones; target, image, error map per pixel
        return dict(bytes=44.0 * n + 192.0 * n * seen + 26.0 * pix, flops=25.0 * pix * walk)
    if kind == "autograd":
        p = case["tiles"] * pix
        # parameters read, every gradient written, colours out and their gradient in
        return dict(bytes=2.0 * 236.0 * n + 24.0 * p, flops=70.0 * p * walk)
    views = case.get("views", 1)
    share = (case["lo"] + case["hi"]) / 2.0 if kind == "views" else case["tiles"]
    p = share * case["rate"] * pix
    touched = seen * (1.0 - (1.0 - min(1.0, share)) ** views)
    # geometry of every Gaussian; parameters and both moments of the touched ones read and written; maps; targets
    return dict(bytes=44.0 * n + 6.0 * 236.0 * n * touched + views * (4.0 * pix + 16.0 * p),
                flops=70.0 * views * p * walk)


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------

def _sh_basis64(d, degree):
    """Real spherical harmonics (Condon-Shortley phase) of unit directions d [N,3], m = -l..l: [N,16]."""
    x, y, z = d.unbind(1)
    pi = math.pi
    c1, c2, c3 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi))
    c4, c5, c6 = math.sqrt(15 / (16 * pi)), math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi))
    c7, c8, c9 = math.sqrt(21 / (32 * pi)), math.sqrt(7 / (16 * pi)), math.sqrt(105 / (16 * pi))
    xx, yy, zz = x * x, y * y, z * z
    Y = [torch.full_like(x, math.sqrt(1 / (4 * pi))), -c1 * y, c1 * z, -c1 * x,
         c2 * x * y, -c2 * y * z, c3 * (2 * zz - xx - yy), -c2 * x * z, c4 * (xx - yy),
         -c5 * y * (3 * xx - yy), c6 * x * y * z, -c7 * y * (4 * zz - xx - yy), c8 * z * (2 * zz - 3 * xx - 3 * yy),
         -c7 * x * (4 * zz - xx - yy), c9 * z * (xx - yy), -c5 * x * (xx - 3 * yy)]
    return torch.stack(Y[:(degree + 1) ** 2], 1)


def _project64(p, cam, degree):
    """EWA projection and SH colour of the 3DGS model: a row (x, y, a, b, c, opacity, r, g, b) per Gaussian,
    and (depth, radius) without gradients (radius 0 where culled)."""
    V = torch.tensor(np.asarray(cam["viewmat"], np.float64).reshape(4, 4), device="cuda")
    R, t = V[:3, :3], V[:3, 3]
    fx, fy, W, H = cam["fx"], cam["fy"], cam["width"], cam["height"]
    pc = p["means"] @ R.T + t
    z = pc[:, 2]
    front = z > cam["znear"]
    z = torch.where(front, z, torch.ones_like(z))
    q = p["quats"] / p["quats"].norm(dim=1, keepdim=True)
    w, x, y, k = q.unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y),
                      2 * (x * y + w * k), 1 - 2 * (x * x + k * k), 2 * (y * k - w * x),
                      2 * (x * k - w * y), 2 * (y * k + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    M = Rq * torch.exp(p["log_scales"])[:, None, :]
    lx, ly = 1.3 * 0.5 * W / fx, 1.3 * 0.5 * H / fy
    tx, ty = (pc[:, 0] / z).clamp(-lx, lx), (pc[:, 1] / z).clamp(-ly, ly)
    zero = torch.zeros_like(z)
    J = torch.stack([fx / z, zero, -fx * tx / z, zero, fy / z, -fy * ty / z], 1).view(-1, 2, 3)
    U = (J @ R) @ M
    A = (U[:, 0] * U[:, 0]).sum(1) + 0.3
    Bc = (U[:, 0] * U[:, 1]).sum(1)
    C = (U[:, 1] * U[:, 1]).sum(1) + 0.3
    det = A * C - Bc * Bc
    eye = -R.T @ t
    d = p["means"] - eye
    d = d / d.norm(dim=1, keepdim=True)
    Y = _sh_basis64(d, degree)
    rgb = (torch.einsum("nk,nkc->nc", Y, p["sh"][:, :Y.shape[1]]) + 0.5).clamp_min(0.0)
    table = torch.cat([torch.stack([fx * pc[:, 0] / z + cam["cx"], fy * pc[:, 1] / z + cam["cy"], C / det, -Bc / det,
                                    A / det, torch.sigmoid(p["opacity_logits"])], 1), rgb], 1)
    with torch.no_grad():
        mid = 0.5 * (A + C)
        lam = mid + torch.sqrt((mid * mid - det).clamp_min(0.1))
        radius = torch.where(front & (det > 0), torch.ceil(3.0 * torch.sqrt(lam)), torch.zeros_like(z))
    return table, z.detach(), radius


def _tile_lists64(table, depth, radius, cam, active):
    """Ids of every active tile's splats in depth order, concatenated, and each tile's offsets."""
    tx_n, ty_n = (cam["width"] + 15) // 16, (cam["height"] + 15) // 16
    rank = torch.full((tx_n * ty_n,), -1, dtype=torch.long, device="cuda")
    rank[torch.tensor(active, device="cuda")] = torch.arange(len(active), device="cuda")
    ids = torch.nonzero(radius > 0).reshape(-1)
    ids = ids[torch.argsort(depth[ids].float(), stable=True)]
    xy, r = table[ids, :2].float(), radius[ids].float()

    def span(c, m):
        return (torch.floor((c - r) / 16).clamp(0, m).long(), (torch.floor((c + r) / 16) + 1).clamp(0, m).long())
    x0, x1 = span(xy[:, 0], tx_n)
    y0, y1 = span(xy[:, 1], ty_n)
    w = x1 - x0
    area = w * (y1 - y0)
    of = torch.repeat_interleave(torch.arange(ids.numel(), device="cuda"), area)
    rem = torch.arange(of.numel(), device="cuda") - (torch.cumsum(area, 0) - area)[of]
    rk = rank[(y0[of] + rem // w[of]) * tx_n + x0[of] + rem % w[of]]
    of, rk = of[rk >= 0], rk[rk >= 0]
    o = torch.argsort(rk, stable=True)
    off = torch.zeros(len(active) + 1, dtype=torch.long, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(rk, minlength=len(active)), 0)
    return ids[of[o]], off.tolist()


def _composite64(t, x, y):
    """Colours of a tile's pixels from its splats' rows t [L,9] in order (black background), and which splats
    each pixel blends."""
    dx = x[:, None] + 0.5 - t[None, :, 0]
    dy = y[:, None] + 0.5 - t[None, :, 1]
    power = -0.5 * (t[:, 2] * dx * dx + t[:, 4] * dy * dy) - t[:, 3] * dx * dy
    alpha = (t[:, 5] * torch.exp(power)).clamp(max=0.99)
    alpha = torch.where((power <= 0) & (alpha >= 1.0 / 255.0), alpha, torch.zeros_like(alpha))
    after = torch.cumprod(1.0 - alpha, 1)
    use = (after.detach() >= 1e-4) & (alpha.detach() > 0)
    before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
    return (torch.where(use, before * alpha, torch.zeros_like(alpha))) @ t[:, 6:9], use


def _render64(scene, cam, degree, active, loss_of=None):
    """Colours of the active tiles' pixels; with loss_of(rank, x, y, rgb), the gradients of the summed losses with
    respect to the parameters and the mask of the Gaussians that a pixel blended."""
    p = {k: v.double().requires_grad_(loss_of is not None) for k, v in scene.items()}
    with torch.set_grad_enabled(loss_of is not None):
        table, depth, radius = _project64(p, cam, degree)
    rows = table.detach()
    ids, off = _tile_lists64(rows, depth, radius, cam, active)
    grad, touched = torch.zeros_like(rows), torch.zeros(rows.shape[0], dtype=torch.bool, device="cuda")
    out = []
    for k, tile in enumerate(active):
        x, y = _tile_pixels(tile, cam["width"], cam["height"])
        i = ids[off[k]:off[k + 1]]
        if i.numel() == 0:
            out.append(torch.zeros(x.numel(), 3, dtype=torch.float64, device="cuda"))
            continue
        t = rows[i].requires_grad_(loss_of is not None)
        with torch.set_grad_enabled(loss_of is not None):
            rgb, use = _composite64(t, x, y)
        if loss_of is not None:
            grad[i] += torch.autograd.grad(loss_of(k, x, y, rgb), t)[0]
            touched[i] |= use.any(0)
        out.append(rgb.detach())
    rgb = torch.cat(out)
    if loss_of is None:
        return rgb
    got = torch.autograd.grad(table, [p[k] for k in FIELDS], grad)
    return rgb, dict(zip(FIELDS, got)), touched


def _tile_loss64(x, y, n_pixels, n_tiles, structure):
    """One tile's share of the sparse loss: Charbonnier L1 and the balanced structure term of predictions x."""
    d = x - y
    l1 = torch.sqrt(d * d + float(np.float32(1e-3)) ** 2)
    mx, my = x.mean(0), y.mean(0)
    vx, vy, cv = ((x - mx) ** 2).mean(0), ((y - my) ** 2).mean(0), ((x - mx) * (y - my)).mean(0)
    if structure == "ncc":
        s = cv / torch.sqrt(vx * vy + 1e-8)
    else:
        s = (2 * mx * my + 1e-4) * (2 * cv + 9e-4) / ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4))
    gs = torch.autograd.grad(s.sum(), x, retain_graph=True)[0]
    mean = lambda g: g.detach().abs().sum(1).mean()  # noqa: E731
    lam = (mean(d / l1) / (x.shape[0] * mean(gs) + 1e-8)).clamp(0.0, 1.0)
    return l1.sum() / n_pixels + lam * (1.0 - s.mean()) / n_tiles


def _update64(case, scene, seed, grads, touched):
    """The late-phase hybrid step (modes 0 and 1) of the touched Gaussians."""
    m0, v0 = _moments(scene, seed)
    o = _config(case).opt
    lr = dict(means=o.lr_means, log_scales=o.lr_scales, quats=o.lr_quats, opacity_logits=o.lr_opacity)
    b1, b2 = o.beta1, o.beta2
    out = dict(params={}, m={}, v={})
    for k in FIELDS:
        p, g = scene[k].double(), grads[k]
        on = touched.view([-1] + [1] * (p.dim() - 1))
        m = torch.where(on, b1 * m0[k].double() + (1 - b1) * g, m0[k].double())
        v = torch.where(on, b2 * v0[k].double() + (1 - b2) * g * g, v0[k].double())
        adam = -(m / (1 - b1 ** STEP_LATE)) / (torch.sqrt(v / (1 - b2 ** STEP_LATE)) + o.eps_adam)
        lm = -m / (g * g + torch.sqrt(v) + o.eps_lm)
        if k == "sh":
            dc = torch.zeros_like(p)
            dc[:, 0] = 1.0
            d = dc * o.lr_sh_dc * (lm if o.mode == 1 else adam) + (1 - dc) * o.lr_sh_rest * adam
        else:
            d = lr[k] * (lm if o.mode == 1 else adam)
        out["params"][k] = torch.where(on, p + d, p)
        out["m"][k], out["v"][k] = m, v
    return out


def _bf16(x):
    return x.float().bfloat16().double()


def _mlp64(case, seed):
    """Forward and, for training, gradient and Adam step of the network, rounding where it stores 16-bit values."""
    s = _prepare_mlp(case, seed)
    mlp = s["mlp"]
    ends = np.cumsum([128 * 16, 128, 128 * 128, 128, 128, 1]).tolist()  # W1 | b1 | W2 | b2 | W3 | b3
    sl = {k: slice(a, b) for k, a, b in zip(("W1", "b1", "W2", "b2", "W3", "b3"), [0] + ends, ends)}
    p = mlp.params.double()
    W1, W2, W3 = _bf16(p[sl["W1"]]).view(128, 16), _bf16(p[sl["W2"]]).view(128, 128), _bf16(p[sl["W3"]])
    b1, b2, b3 = p[sl["b1"]], p[sl["b2"]], p[sl["b3"]]
    rows = case["rows"]
    grad, ys = torch.zeros_like(p), []
    for a in range(0, rows, 1 << 18):
        x = _bf16(s["x"][a:a + (1 << 18)])
        h1 = _bf16((x @ W1.T + b1).clamp_min(0.0))
        h2 = _bf16((h1 @ W2.T + b2).clamp_min(0.0))
        y = h2 @ W3 + b3
        ys.append(y)
        if case["kind"] == "predict":
            continue
        dy = (y - s["target"][a:a + (1 << 18)].double()) / rows
        dh2 = _bf16((dy[:, None] * W3) * (h2 > 0))
        dh1 = _bf16((dh2 @ W2) * (h1 > 0))
        for name, g in (("W1", dh1.T @ x), ("b1", dh1.sum(0)), ("W2", dh2.T @ h1), ("b2", dh2.sum(0)),
                        ("W3", dy @ h2), ("b3", dy.sum())):
            grad[sl[name]] += g.reshape(-1)
    if case["kind"] == "predict":
        return dict(y=torch.cat(ys))
    t = STEP_LATE + 1
    m = 0.9 * mlp.m.double() + 0.1 * grad
    v = 0.999 * mlp.v.double() + 0.001 * grad * grad
    step = mlp.lr * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return dict(grads=grad, params=p - step, m=m, v=v)


def exact(case, seed):
    """64-bit outputs.  None for the sampled steps, whose pixels a hash draws and whose state has no closed value
    apart from that draw, and for scenes whose tiles would take too long one by one."""
    kind = case["kind"]
    if kind in ("predict", "train"):
        return _mlp64(case, seed)
    if kind in ("views", "view_draw") or (kind == "step" and (not case["dense"] or case["stats"])):
        return None
    W, H, n = case["width"], case["height"], case["n"]
    tiles = list(range(((W + 15) // 16) * ((H + 15) // 16)))
    scene, cam = _scene(n, seed), _camera(n, W, H)
    if kind == "refresh":
        if len(tiles) > 9000:
            return None
        rgb = _render64(scene, cam, case["sh_degree"], tiles)
        target, error, at = _image(W, H, seed, 2).double(), torch.zeros(H, W, dtype=torch.float64, device="cuda"), 0
        for k in tiles:
            x, y = _tile_pixels(k, W, H)
            error[y, x] = (rgb[at:at + x.numel()] - target[y, x]).abs().sum(1)
            at += x.numel()
        return dict(rgb=rgb, error=error)
    if kind == "autograd":
        tiles = _tile_set(case)
    if len(tiles) > 4000:
        return None
    target = _image(W, H, seed, 2).double()
    pixels = sum(_tile_pixels(k, W, H, "cpu")[0].numel() for k in tiles) if kind == "autograd" else W * H
    if kind == "autograd":
        def loss_of(k, x, y, rgb):
            return ((rgb - target[y, x]) ** 2).sum() / (3.0 * pixels)
        rgb, grads, _ = _render64(scene, cam, case["sh_degree"], tiles, loss_of)
        return dict(rgb=rgb, grads=grads)

    def loss_of(k, x, y, rgb):
        return _tile_loss64(rgb, target[y, x], pixels, len(tiles), case["structure"])
    _, grads, touched = _render64(scene, cam, case["sh_degree"], tiles, loss_of)
    return _update64(case, scene, seed, grads, touched)
