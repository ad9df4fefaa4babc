"""The calls a user of the renderer makes, at the sizes they are made at.

Scenes are the repository's two synthetic performers (inputs.make_shape): a
solid union of 5 ellipsoids (8 basis weights, 30 frames, degree 2) and a
noise-displaced shell around 12 ellipsoids (16 weights, 150 frames, degree 3),
built at any depth.  Coefficients are rounded to BF16 so that BF16 storage
holds them exactly and ``exact`` speaks of the arithmetic alone.

Kinds of case:
  view       one camera frame, rays on the device (viewer, evaluation)
  train      one optimisation step over whole views: forward, MSE and image-gradient loss, adjoint, Adam
  batch      one optimisation step over rays drawn from many views and times
  autograd   the torch.autograd.Function, forward and backward
  compose    several transformed primitives in one frame (mono or stereo)
  slice      a paused moment: time slice of the whole tree, then its frame
  lit        a frame under a spotlight: render, the light's alpha map, its filter, the shading
  edit       painting on the performer: pick, paint, edited render
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2202_06088_gb300 import binding as nv
from paper_2202_06088_gb300 import inputs

DEV = "cuda"
FOV = 40.0
RADIUS = 2.5                      # the cameras' distance from the scene's centre
TAN = math.tan(math.radians(FOV) / 2)
T_STOP = 1e-4
LR, BETA1, BETA2, EPS, STEP = 1e-3, 0.9, 0.999, 1e-8, 100
LAMBDA = 0.1                      # weight of the image-gradient loss
LIGHT = 256                       # the light's alpha map, pixels per side
BLUR = 1.0
GROUND, ALBEDO, R_REF = 0.0, (0.8, 0.8, 0.8), 2.5
SIZES = {"solid": dict(K=8, T=30, degree=2), "shell": dict(K=16, T=150, degree=3)}


def listed():
    return [
        # a thumbnail of a small tree in FP32: the smallest call, launches and latency
        dict(name="view_128", kind="view", scene="solid", depth=6, leaves=20_000, dtype="f32", width=128, height=128),
        # one frame of a full-size performer as a viewer asks for it
        dict(name="view_1080p", kind="view", scene="shell", depth=9, leaves=2_000_000, dtype="bf16", width=1920,
             height=1080),
        # a frame of odd size from the compact storage
        dict(name="view_odd_fp8", kind="view", scene="shell", depth=8, leaves=500_000, dtype="fp8", width=1283,
             height=717),
        # the headline training step: 8 whole views at 8 times
        dict(name="train_8x1080p", kind="train", scene="shell", depth=9, leaves=2_000_000, dtype="bf16", views=8,
             width=1920, height=1080),
        # a data loader's batch on a tree with more leaves than samples per view
        dict(name="batch_262k", kind="batch", scene="solid", depth=8, leaves=1_280_000, dtype="bf16", rays=262_144,
             views=16, order="given"),
        # a large batch on the deepest tree, its rays grouped by the library
        dict(name="batch_1m_deep", kind="batch", scene="shell", depth=10, leaves=2_000_000, dtype="bf16",
             rays=1_048_576, views=32, order="rays"),
        # fitting a small tree through autograd, FP32 throughout
        dict(name="autograd_16k", kind="autograd", scene="solid", depth=6, leaves=20_000, dtype="f32", rays=16_384,
             views=4),
        # eight performers for a headset
        dict(name="compose_stereo", kind="compose", scene="solid", depth=6, leaves=20_000, dtype="bf16", prims=8,
             width=2160, height=2160, eyes=2, mode="sorted"),
        # a small preview of a composition, Algorithm 1 as written
        dict(name="compose_preview", kind="compose", scene="solid", depth=6, leaves=20_000, dtype="f32", prims=3,
             width=640, height=360, eyes=1, mode="alg1"),
        # stepping through time on a paused frame
        dict(name="slice_1080p", kind="slice", scene="shell", depth=9, leaves=2_000_000, dtype="bf16", width=1920,
             height=1080),
        # a lit frame
        dict(name="lit_1080p", kind="lit", scene="shell", depth=9, leaves=2_000_000, dtype="bf16", width=1920,
             height=1080),
        # an editing session's frame
        dict(name="edit_720p", kind="edit", scene="shell", depth=8, leaves=500_000, dtype="bf16", width=1280,
             height=720),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "train", "batch", "batch", "autograd", "compose", "slice", "lit", "edit"])
    scene = "solid" if kind in ("autograd", "compose") else rng.choice(["solid", "shell"])
    c = dict(kind=kind, scene=scene)
    if scene == "solid":
        c["depth"] = rng.choice([5, 6, 7]) if kind in ("autograd", "compose") else rng.choice([6, 7, 8])
        c["leaves"] = int(20_000 * 8.0 ** (c["depth"] - 6))
    else:
        c["depth"] = rng.choice([7, 8, 9])
        c["leaves"] = int({7: 120_000, 8: 500_000, 9: 2_000_000}[c["depth"]] * math.exp(rng.uniform(-0.7, 0.0)))
    c["dtype"] = rng.choice(["f32", "bf16"] if kind == "edit" else ["f32", "bf16", "bf16", "fp8"])
    if kind in ("view", "slice", "lit", "edit"):
        c["height"] = _log_int(rng, 97, 1200)
        c["width"] = max(64, int(c["height"] * rng.uniform(0.8, 1.9)))
    elif kind == "train":
        c["views"] = rng.randint(2, 6)
        c["height"] = _log_int(rng, 240, 1080)
        c["width"] = max(64, int(c["height"] * rng.uniform(1.0, 1.78)))
    elif kind in ("batch", "autograd"):
        c["rays"] = _log_int(rng, 20_000, 500_000) if kind == "batch" else _log_int(rng, 4_000, 130_000)
        c["views"] = rng.randint(2, 32)
        if kind == "batch":
            c["order"] = rng.choice(["given", "rays"])
    else:
        c["prims"] = rng.randint(2, 10)
        c["height"] = _log_int(rng, 200, 2000)
        c["width"] = max(64, int(c["height"] * rng.uniform(0.8, 1.8)))
        c["eyes"] = rng.choice([1, 2])
        c["mode"] = rng.choice(["sorted", "sorted", "alg1"])
    return c


# ----------------------------------------------------------------------------
# Scenes
# ----------------------------------------------------------------------------

def _field(shape, scale, p):
    """Approximate signed distance of points p [n, 3] to the shape."""
    def t64(a):
        return torch.as_tensor(np.asarray(a), dtype=torch.float64, device=DEV)
    f = torch.full((p.shape[0],), math.inf, dtype=torch.float64, device=DEV)
    for c, a, R in zip(shape.centers, shape.axes * scale, shape.rots):
        r = (((p - t64(c)) @ t64(R)) / t64(a)).square().sum(1).sqrt()
        f = torch.minimum(f, (r - 1.0) * float(a.min()))
    if shape.noise_amp:
        s = torch.zeros_like(f)
        for w, ph, a in zip(shape.noise_w, shape.noise_phase, shape.noise_a):
            s += float(a) * torch.sin(p @ t64(w) + float(ph))
        f = f + shape.noise_amp * s / float(shape.noise_a.sum())
    return f


def _cells(shape, depth, scale=1.0, h=None):
    """Morton keys of the occupied finest cells, ascending: the field at the
    cell's centre is <= 0 (h None) or within h of 0."""
    keys, lip = torch.zeros(1, dtype=torch.int64, device=DEV), shape.lipschitz()
    for L in range(1, depth + 1):
        keys = ((keys[:, None] << 3) | torch.arange(8, device=DEV)).reshape(-1)
        r = 0.5 * math.sqrt(3.0) * (2.0 ** -L - 2.0 ** -depth)
        keep = []
        for part in keys.split(1 << 22):
            f = _field(shape, scale, (_coords(part, L).double() + 0.5) * 2.0 ** -L)
            keep.append((f - lip * r <= 0.0) if h is None else (f.abs() - lip * r < h))
        keys = keys[torch.cat(keep)]
    return keys


def _coords(keys, depth):
    c = torch.zeros(keys.numel(), 3, dtype=torch.int64, device=DEV)
    for b in range(depth):
        for a in range(3):
            c[:, a] |= ((keys >> (3 * b + 2 - a)) & 1) << b
    return c


def _child_table(keys, depth):
    """Breadth-first child table of the tree whose leaves are the finest cells `keys`."""
    levels = [torch.unique(keys >> (3 * (depth - L))) for L in range(depth)]
    base = np.cumsum([0] + [k.numel() for k in levels])
    child = torch.full((int(base[-1]), 8), -1, dtype=torch.int64, device=DEV)
    for L, nodes in enumerate(levels):
        below = levels[L + 1] if L + 1 < depth else keys
        want = ((nodes[:, None] << 3) | torch.arange(8, device=DEV)).reshape(-1)
        at = torch.searchsorted(below, want).clamp_(max=below.numel() - 1)
        entry = at + int(base[L + 1]) if L + 1 < depth else at | 0x80000000
        child[base[L]:base[L + 1]] = torch.where(below[at] == want, entry, -1).reshape(-1, 8)
    return (child & 0xFFFFFFFF).cpu().numpy().astype(np.uint32).reshape(-1)


@functools.lru_cache(maxsize=6)
def _scene(scene, depth, leaves):
    """Host tree, device coefficients [n, 2K + 3 N_h] and the dense grid of leaf ids."""
    size = SIZES[scene]
    K, T, degree = size["K"], size["T"], size["degree"]
    rng = np.random.default_rng(1234 + depth)
    if scene == "solid":
        shape = inputs.make_shape(rng, 5, 0.3, 0.7, 0.08, 0.2)
        lo, hi = 0.25, 4.0
        for _ in range(14):
            mid = math.sqrt(lo * hi)
            lo, hi = (mid, hi) if _cells(shape, 6, mid).numel() < leaves / 8.0 ** (depth - 6) else (lo, mid)
        keys = _cells(shape, depth, math.sqrt(lo * hi))
    else:
        shape, h = inputs.make_shape(rng, 12, 0.25, 0.75, 0.08, 0.22, noise_amp=0.02), 2.0 ** (1 - depth)
        for _ in range(2):
            h *= leaves / max(_cells(shape, depth, h=h).numel(), 1)
        keys = _cells(shape, depth, h=h)
    n, nh = keys.numel(), inputs.n_hh(degree)
    g = torch.Generator(DEV).manual_seed(99 + depth)
    w = torch.randn(n, 2 * K + 3 * nh, device=DEV, generator=g)
    w[:, :K] = torch.nn.functional.softplus(w[:, :K])
    w[:, 2 * K:] *= 0.3
    w = w.bfloat16().float()
    a = inputs.smooth_curves(rng, T, K)
    a *= 30.0 / (K * max(float(np.abs(a).mean()), 1e-6) * 0.8065786)
    b = (2.0 * inputs.smooth_curves(rng, T, K) - 1.0) * (2.0 / math.sqrt(K))
    cells = _coords(keys, depth)
    st = inputs.TreeStructure(depth, _child_table(keys, depth), np.full(n, depth, np.int32),
                              cells.int().cpu().numpy())
    planes = w.t().contiguous().cpu().numpy()
    host = inputs.VOctree(st, K, T, degree, planes[:K], planes[K:2 * K], planes[2 * K:].reshape(3, nh, n),
                          a.astype(np.float32), b.astype(np.float32))
    grid = torch.full((1 << 3 * depth,), -1, dtype=torch.int32, device=DEV)
    N = 1 << depth
    grid[(cells[:, 0] * N + cells[:, 1]) * N + cells[:, 2]] = torch.arange(n, dtype=torch.int32, device=DEV)
    return SimpleNamespace(host=host, w=w, grid=grid, depth=depth, K=K, T=T, degree=degree, nh=nh, n=n,
                           A=torch.as_tensor(host.basis_A, device=DEV).double(),
                           B=torch.as_tensor(host.basis_B, device=DEV).double())


def _scene_of(c):
    return _scene(c["scene"], c["depth"], c["leaves"])


@functools.lru_cache(maxsize=6)
def _shared_tree(scene, depth, leaves, dtype):
    """The handle that a program which only renders keeps."""
    return nv.Tree(_scene(scene, depth, leaves).host, dtype)


def _tree_of(c):
    return _shared_tree(c["scene"], c["depth"], c["leaves"], c["dtype"])


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------

def _pixel_dirs(cam, pixels):
    """Unit directions [3, n] through the centres of row-major pixels (FP64)."""
    px, py = (pixels % cam.width).double(), (pixels // cam.width).double()
    th = math.tan(math.radians(cam.fov_y_deg) / 2.0)
    sx = (2.0 * (px + 0.5) / cam.width - 1.0) * th * (cam.width / cam.height)
    sy = (1.0 - 2.0 * (py + 0.5) / cam.height) * th
    f, r, u = (torch.as_tensor(np.asarray(v), device=DEV)[:, None] for v in (cam.forward, cam.right, cam.up))
    d = f + r * sx + u * sy
    return d / d.norm(dim=0, keepdim=True)


def _tiled_pixels(width, height):
    """Row-major pixels listed by 8 x 4 tiles (a 32-ray packet per tile)."""
    p = torch.arange(width * height, device=DEV)
    x, y = p % width, p // width
    key = ((y // 4) * ((width + 7) // 8) + x // 8) * 32 + (y % 4) * 8 + x % 8
    return torch.argsort(key)


def _view_rays(cams, times):
    """Rays of whole views, tile by tile, and the ray of each pixel [views, height, width]."""
    o, d, t, rop, first = [], [], [], [], 0
    for cam, time in zip(cams, times):
        pix = _tiled_pixels(cam.width, cam.height)
        d.append(_pixel_dirs(cam, pix))
        o.append(torch.as_tensor(np.asarray(cam.eye), device=DEV)[:, None].expand(3, pix.numel()))
        t.append(torch.full((pix.numel(),), float(time), device=DEV))
        m = torch.empty(pix.numel(), dtype=torch.int32, device=DEV)
        m[pix] = torch.arange(first, first + pix.numel(), dtype=torch.int32, device=DEV)
        rop.append(m.view(1, cam.height, cam.width))
        first += pix.numel()
    return torch.cat(o, 1).float(), torch.cat(d, 1).float(), torch.cat(t), torch.cat(rop)


def _batch_rays(seed, n, views, side=512):
    """Rays drawn uniformly over views, 16 times and pixels, in the order drawn."""
    g = torch.Generator(DEV).manual_seed(seed)
    view = torch.randint(views, (n,), device=DEV, generator=g)
    pix = torch.randint(side * side, (n,), device=DEV, generator=g)
    t = torch.randint(16, (n,), device=DEV, generator=g).float() / 15.0
    o, d = torch.empty(3, n, device=DEV), torch.empty(3, n, device=DEV)
    for v, cam in enumerate(inputs.sphere_cameras(seed, views, RADIUS, side, side)):
        at = torch.nonzero(view == v).reshape(-1)
        d[:, at] = _pixel_dirs(cam, pix[at]).float()
        o[:, at] = torch.as_tensor(np.asarray(cam.eye), device=DEV).float()[:, None]
    return o, d, t


def _inputs(c, seed):
    """What both prepare() and exact() start from, made from the seed alone."""
    rng = np.random.default_rng(seed)
    g = torch.Generator(DEV).manual_seed(seed + 7)
    s = SimpleNamespace(kind=c["kind"])
    if c["kind"] in ("view", "slice", "lit", "edit", "train"):
        s.views = c.get("views", 1)
        cams = inputs.sphere_cameras(seed, s.views, RADIUS, c["width"], c["height"])
        s.times = rng.uniform(0.0, 1.0, s.views).astype(np.float32)
        s.o, s.d, s.t, s.ray_of_pixel = _view_rays(cams, s.times)
    elif c["kind"] in ("batch", "autograd"):
        s.o, s.d, s.t = _batch_rays(seed, c["rays"], c["views"])
    else:
        s.prims = inputs.config4_primitives(c["prims"], T=SIZES[c["scene"]]["T"], seed=seed)
        v = rng.standard_normal(3)
        eye = 8.0 * v / np.linalg.norm(v)
        mid = inputs.look_at(eye, np.zeros(3), c["width"], c["height"])
        side = [0.0] if c["eyes"] == 1 else [-0.032, 0.032]
        cams = [inputs.look_at(eye + x * mid.right, np.zeros(3), c["width"], c["height"]) for x in side]
        s.times = np.full(c["eyes"], rng.uniform(0.0, 1.0), np.float32)
        s.o, s.d, s.t, _ = _view_rays(cams, s.times)
    s.n = s.t.numel()
    if c["kind"] in ("train", "batch"):
        s.target = 0.5 * torch.rand(s.n, 3, device=DEV, generator=g)
        # optimizer state of a run under way: gradients of the size these losses give
        shape = (_scene_of(c).n, _scene_of(c).w.shape[1])
        size = 0.1 / s.n
        s.m = torch.randn(shape, device=DEV, generator=g) * size
        s.v = torch.rand(shape, device=DEV, generator=g).add_(0.1) * size * size
    elif c["kind"] == "autograd":
        s.w = _scene_of(c).w + 0.05 * torch.randn(_scene_of(c).w.shape, device=DEV, generator=g)
        s.g_rgb = torch.randn(s.n, 3, device=DEV, generator=g) / s.n
        s.g_alpha = torch.randn(s.n, device=DEV, generator=g) / s.n
    elif c["kind"] == "lit":
        u = rng.standard_normal(2)
        eye = np.array([0.5 + 0.6 * u[0] / np.hypot(*u), 0.5 + 0.6 * u[1] / np.hypot(*u), 2.6])
        s.light = inputs.look_at(eye, (0.5, 0.5, 0.5), LIGHT, LIGHT)
        s.lo, s.ld, s.lt, s.light_map = _view_rays([s.light], s.times)
    elif c["kind"] == "edit":
        s.color = torch.rand(s.n, 3, device=DEV, generator=g)
    return s


def _padded(x, stride):
    return torch.nn.functional.pad(x, (0, stride - x.shape[1]))


def prepare(case, seed):
    c = case
    s = _inputs(c, seed)
    s.rays = nv.DeviceRays(s.o, s.d, s.t)
    s.time = float(s.t[0])
    if c["kind"] in ("train", "batch"):
        s.tree = nv.Tree(_scene_of(c).host, c["dtype"], with_optimizer=True)
        m, v = s.tree.adam_state()
        m.copy_(_padded(s.m, m.shape[1]))
        v.copy_(_padded(s.v, v.shape[1]))
        del s.m, s.v
        if c.get("order") == "rays":
            s.tree.set_packet_order(nv.ORDER_BY_RAY)
        # a log with room for every segment; whole views take the leaf-major adjoint
        per_ray = 64 if c["kind"] == "train" else 256
        s.out = nv.alloc_out(s.n, log_bytes_per_ray=per_ray)
        if c["kind"] == "train":
            s.tree.reserve_adjoint(s.n * per_ray // 8)
        s.grad, s.touched = s.tree.new_grad(), s.tree.new_touched()
        s.grad_rgb, s.loss = torch.empty(s.n, 3, device=DEV), torch.zeros(1, device=DEV)
    elif c["kind"] == "autograd":
        s.tree = nv.Tree(_scene_of(c).host, c["dtype"])
        s.coeffs = _padded(s.w, s.tree.info.rec_stride_f32).requires_grad_()
    elif c["kind"] == "compose":
        s.trees = [_tree_of(c)] * c["prims"]
        s.xf = np.stack([p.transform for p in s.prims])
        s.off = [p.time_offset for p in s.prims]
        s.tint = np.stack([p.tint for p in s.prims])
        s.mode = c["mode"]
        s.out = {k: torch.empty(s.n, 3, device=DEV) if k == "rgb" else torch.empty(s.n, device=DEV)
                 for k in ("rgb", "alpha", "depth")}
    else:
        s.tree = _tree_of(c)
        s.out = nv.alloc_out(s.n)
        if c["kind"] == "slice":
            s.slice = torch.zeros(s.tree.n_leaves, nv.slice_stride(s.tree.info.hh_degree), device=DEV)
        elif c["kind"] == "lit":
            s.light_rays = nv.DeviceRays(s.lo, s.ld, s.lt)
            s.pixel = s.light_map.reshape(-1).long()
        elif c["kind"] == "edit":
            s.blank = nv.new_edits(s.tree)
    return s


def _image(out):
    return {k: out[k] for k in ("rgb", "alpha", "depth", "tau", "nseg") if k in out}


def run(s):
    if s.kind == "view":
        return _image(nv.neuvv_render(s.tree, s.rays, out=s.out))
    if s.kind in ("train", "batch"):
        nv.neuvv_render(s.tree, s.rays, kernel="packet", out=s.out)
        s.loss.zero_()
        nv.neuvv_mse_grad(s.out["rgb"], s.target, scale=1.0 / s.n, grad=s.grad_rgb, loss=s.loss)
        if s.kind == "train":
            nv.neuvv_grad_loss(s.out["rgb"], s.target, s.ray_of_pixel, LAMBDA / s.n, s.grad_rgb, s.loss)
        nv.neuvv_render_backward_adam(s.tree, s.rays, s.out, s.grad_rgb, None, s.grad, s.touched, lr=LR, beta1=BETA1,
                                      beta2=BETA2, eps=EPS, step=STEP)
        m, v = s.tree.adam_state()
        return dict(_image(s.out), loss=s.loss, master=s.tree.master(), m=m, v=v, storage=s.tree.storage())
    if s.kind == "autograd":
        s.coeffs.grad = None
        rgb, alpha, depth = nv.render_differentiable(s.coeffs, s.tree, s.rays)
        torch.autograd.backward([rgb, alpha], [s.g_rgb, s.g_alpha])
        return {"rgb": rgb, "alpha": alpha, "depth": depth, "grad": s.coeffs.grad}
    if s.kind == "compose":
        return nv.neuvv_compose(s.trees, s.xf, s.off, s.tint, s.rays, mode=s.mode, out=s.out)
    if s.kind == "slice":
        nv.neuvv_slice(s.tree, s.time, out=s.slice)
        return dict(_image(nv.neuvv_render_slice(s.tree, s.slice, s.rays, out=s.out)), slice=s.slice)
    if s.kind == "lit":
        la = nv.neuvv_render_alpha(s.tree, s.light_rays)["alpha"]
        shadow = nv.neuvv_gaussian_blur(la[s.pixel].view(1, LIGHT, LIGHT), BLUR)
        out = nv.neuvv_render(s.tree, s.rays, out=s.out)
        lit = nv.neuvv_spotlight(s.rays, out, s.light, shadow[0], GROUND, ALBEDO, R_REF)
        return dict(_image(out), lit=lit, shadow=shadow)
    leaf = nv.neuvv_pick(s.tree, s.rays)
    edits = nv.neuvv_paint(s.tree, leaf, s.color, -1.0, 0.0, s.blank.clone())
    return dict(_image(nv.neuvv_render_edit(s.tree, s.rays, edits, beta=0.7, out=s.out)), leaf=leaf, edits=edits)


# ----------------------------------------------------------------------------
# Work of one pass
# ----------------------------------------------------------------------------

def work(case):
    """Segments from the mean projected area of a cell (1.5 side^2) and the
    rays per unit area at the scene; leaves touched as in a random cover."""
    c, k = case, SIZES[case["scene"]]
    K, nh = k["K"], inputs.n_hh(k["degree"])
    P = (k["degree"] + 1) * (k["degree"] + 2) // 2
    length = 2 * K + 3 * nh
    rec = {"f32": 4 * length, "bf16": 2 * length, "fp8": length + 12}[c["dtype"]]
    h = 2.0 ** -c["depth"]
    if c["kind"] in ("batch", "autograd"):
        n = c["rays"]
        samples = n * c["leaves"] * 1.5 * h * h / (2 * RADIUS * TAN) ** 2
    elif c["kind"] == "compose":
        n = c["width"] * c["height"] * c["eyes"]
        samples = c["eyes"] * c["prims"] * c["leaves"] * 1.5 * h * h * (c["height"] / (2 * 8.0 * TAN)) ** 2
    else:
        views = c.get("views", 1)
        n = c["width"] * c["height"] * views
        samples = views * c["leaves"] * 1.5 * h * h * (c["height"] / (2 * RADIUS * TAN)) ** 2
    touched = c["leaves"] * -math.expm1(-samples / c["leaves"])
    per_sample = 4 * K + 4 * P + 6 * (nh + P) + 20
    bytes_, flops = n * (28 + 28) + touched * rec, samples * per_sample
    if c["kind"] in ("train", "batch", "autograd"):
        bytes_ += n * (28 + 20 + 12) + touched * rec      # the adjoint's rays, saved state and records
        flops *= 3
        if c["kind"] == "autograd":
            bytes_ += c["leaves"] * length * 4 * 3        # coefficients into the tree, gradient out
        else:
            bytes_ += n * 36 + touched * (24 * length + rec)  # loss; master and moments in and out, storage out
            flops += touched * length * 12
    elif c["kind"] == "slice":
        row = 4 * (1 + 3 * (k["degree"] + 1) ** 2)
        bytes_ += c["leaves"] * (rec + row) + touched * (row - rec)
        flops += c["leaves"] * (4 * K + 6 * nh)
    elif c["kind"] == "lit":
        bytes_ += n * 24 + LIGHT * LIGHT * 64
    elif c["kind"] == "edit":
        bytes_ += n * (28 + 4 + 12) + touched * (4 * K + 32)
    return {"bytes": bytes_, "flops": flops}


# ----------------------------------------------------------------------------
# The same results in 64 bits, by plain tensor operations
# ----------------------------------------------------------------------------

def _segments(sc, o, d):
    """Occupied cells on rays o + s d (FP64 [n, 3], d unit) of the unit cube:
    (ray, leaf, t0, t1), by ray and front to back."""
    N, n = 1 << sc.depth, o.shape[0]
    inv = torch.where(d != 0, 1.0 / d, math.inf)
    near = torch.where(d > 0, -o * inv, torch.where(d < 0, (1.0 - o) * inv, -math.inf))
    far = torch.where(d > 0, (1.0 - o) * inv, torch.where(d < 0, -o * inv, math.inf))
    inside = ((d != 0) | ((o >= 0) & (o <= 1))).all(1)
    t0, t1 = near.amax(1).clamp_min(0.0), far.amin(1)
    at = torch.nonzero(inside & (t0 < t1)).reshape(-1)
    ray, o, d, inv, near, t = at, o[at] * N, d[at] * N, inv[at] / N, near[at], t0[at]
    p = o + t[:, None] * d
    cell = torch.where(d < 0, p.ceil() - 1, p.floor()).clamp_(0, N - 1)
    entry = (near == t[:, None])
    cell = torch.where(entry, torch.where(d < 0, N - 1.0, 0.0), cell)
    found = []
    while ray.numel():
        plane = cell + (d > 0)
        tx = torch.where(d != 0, (plane - o) * inv, math.inf)
        ax = torch.where(tx[:, 1] < tx[:, 0], 1, 0)
        te = torch.minimum(tx[:, 0], tx[:, 1])
        ax = torch.where(tx[:, 2] < te, 2, ax)
        te = torch.minimum(te, tx[:, 2])
        c = cell.long()
        leaf = sc.grid[(c[:, 0] * N + c[:, 1]) * N + c[:, 2]]
        hit = torch.nonzero((leaf >= 0) & (te > t)).reshape(-1)
        found.append((ray[hit], leaf[hit], t[hit], te[hit]))
        t = torch.maximum(t, te)
        step = torch.nn.functional.one_hot(ax, 3) * torch.sign(d)
        cell = cell + step
        live = ((cell >= 0) & (cell < N)).all(1)
        if not bool(live.all()):
            ray, o, d, inv, t, cell = ray[live], o[live], d[live], inv[live], t[live], cell[live]
    if not found:
        z = torch.zeros(0, dtype=torch.int64, device=DEV)
        return z, z, z.double(), z.double()
    ray, leaf, t0, t1 = (torch.cat(x) for x in zip(*found))
    by = torch.argsort(ray, stable=True)
    return ray[by], leaf[by].long(), t0[by], t1[by]


def _harmonics(degree, d):
    x, y, z = d.unbind(1)
    Y = [torch.full_like(x, math.sqrt(1 / (4 * math.pi)))]
    if degree >= 1:
        k = math.sqrt(3 / (4 * math.pi))
        Y += [k * y, k * z, k * x]
    if degree >= 2:
        k = math.sqrt(15 / (4 * math.pi))
        Y += [k * x * y, k * y * z, math.sqrt(5 / (16 * math.pi)) * (3 * z * z - 1), k * x * z, 0.5 * k * (x * x - y * y)]
    if degree >= 3:
        a, b, e = math.sqrt(35 / (32 * math.pi)), math.sqrt(105 / (4 * math.pi)), math.sqrt(21 / (32 * math.pi))
        Y += [a * y * (3 * x * x - y * y), b * x * y * z, e * y * (5 * z * z - 1),
              math.sqrt(7 / (16 * math.pi)) * z * (5 * z * z - 3), e * x * (5 * z * z - 1),
              0.5 * b * z * (x * x - y * y), a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _gegenbauer(lam, k, x):
    if k < 0:
        return torch.zeros_like(x)
    c0, c1 = torch.ones_like(x), 2.0 * lam * x
    if k == 0:
        return c0
    for j in range(2, k + 1):
        c0, c1 = c1, (2.0 * x * (j + lam - 1) * c1 - (j + 2 * lam - 2) * c0) / j
    return c1


def _radial(degree, g):
    """R_nl(g) and dR_nl/dg, and for each harmonic its (n, l) and (l, m) column."""
    s, x = torch.sin(g), torch.cos(g)
    R, D, col, lm = [], [], [], []
    for n in range(degree + 1):
        for l in range(n + 1):
            a = 2.0 ** l * math.factorial(l) * math.sqrt(
                2.0 * (n + 1) * math.factorial(n - l) / (math.pi * math.factorial(n + l + 1)))
            c = _gegenbauer(l + 1, n - l, x)
            R.append(a * s ** l * c)
            low = l * s ** (l - 1) * x * c if l else torch.zeros_like(x)
            D.append(a * (low - s ** (l + 1) * 2.0 * (l + 1) * _gegenbauer(l + 2, n - l - 1, x)))
            for m in range(-l, l + 1):
                col.append(len(R) - 1)
                lm.append(l * l + l + m)
    return torch.stack(R, 1), torch.stack(D, 1), col, lm


def _rows(sc, u):
    u = u.clamp(0, sc.T - 1)
    f0 = u.floor().long()
    f1, fr = (f0 + 1).clamp_max(sc.T - 1), (u - f0)[:, None]
    return (1 - fr) * sc.A[f0] + fr * sc.A[f1], (1 - fr) * sc.B[f0] + fr * sc.B[f1]


def _shade(sc, w, leaf, u, d):
    """Per-sample values of leaves seen along unit d at frame coordinate u."""
    K, r = sc.K, w[leaf].double()
    a, b = _rows(sc, u)
    pre = (a * r[:, :K]).sum(1)
    sg = torch.sigmoid((b * r[:, K:2 * K]).sum(1))
    R, D, col, lm = _radial(sc.degree, math.pi * sg)
    Y = _harmonics(sc.degree, d)
    part = r[:, 2 * K:].view(-1, 3, sc.nh) * Y[:, None, lm]
    z, dz = (part * R[:, None, col]).sum(2), (part * D[:, None, col]).sum(2)
    return SimpleNamespace(pre=pre, sigma=pre.clamp_min(0.0), col=torch.sigmoid(z), sg=sg, dz=dz, a=a, b=b,
                           H=(Y[:, lm] * R[:, col]))


CHUNK = 1 << 20


def _render(sc, w, o, d, u, scale=None, edit=None):
    """Images and the composited segments of rays (FP64 [n, 3], any length of d)."""
    n = o.shape[0]
    dn = d / d.norm(dim=1, keepdim=True)
    ray, leaf, t0, t1 = _segments(sc, o, dn)
    dt = t1 - t0
    sig, col = [], []
    for at in torch.arange(ray.numel(), device=DEV).split(CHUNK):
        v = _shade(sc, w, leaf[at], u[ray[at]], dn[ray[at]])
        sig.append(v.sigma)
        col.append(v.col)
    sig = torch.cat(sig) if sig else dt
    col = torch.cat(col) if col else dt.new_zeros(0, 3)
    if edit is not None:
        e = edit[leaf]
        on = e[:, 4] <= 1.0
        col = torch.where(on[:, None], col + 0.7 * (e[:, :3] - col), col)
    sd = sig * dt
    run_, first = sd.cumsum(0), torch.searchsorted(ray, torch.arange(n, device=DEV))
    lead = torch.cat([sd.new_zeros(1), run_])
    before = (lead[:-1] - lead[first][ray]).clamp_min(0.0)
    keep = before <= -math.log(T_STOP)
    ray, leaf, t0, dt, sd, col, before, sig = (x[keep] for x in (ray, leaf, t0, dt, sd, col, before, sig))
    wgt = torch.exp(-before) * -torch.expm1(-sd)

    def total(x):
        return torch.zeros((n,) + x.shape[1:], dtype=torch.float64, device=DEV).index_add_(0, ray, x)
    rgb, alpha, tau = total(wgt[:, None] * col), total(wgt), total(sd)
    mid = t0 + 0.5 * dt
    if scale is not None:
        mid = mid * scale[ray]
    depth = torch.where(alpha >= 1e-4, total(wgt * mid) / alpha, math.inf)
    return SimpleNamespace(rgb=rgb, alpha=alpha, depth=depth, tau=tau, ray=ray, leaf=leaf, dt=dt, sd=sd, col=col,
                           before=before, sig=sig, w=wgt, dn=dn)


def _adjoint(sc, w, f, u, g, g_alpha):
    """Gradient of the coefficients and the leaves that a composited sample reached."""
    grad, n = torch.zeros(w.shape, dtype=torch.float64, device=DEV), f.rgb.shape[0]
    wc = f.w[:, None] * f.col
    lead = torch.cat([wc.new_zeros(1, 3), wc.cumsum(0)])
    first = torch.searchsorted(f.ray, torch.arange(n, device=DEV))
    after = f.rgb[f.ray] - (lead[1:] - lead[first][f.ray])
    left = torch.exp(-f.before - f.sd)
    dsig = (g[f.ray] * (left[:, None] * f.col - after)).sum(1)
    if g_alpha is not None:
        dsig = dsig + g_alpha[f.ray] * torch.exp(-f.tau[f.ray])
    dsig = torch.where(f.sig > 0, dsig * f.dt, 0.0)
    for at in torch.arange(f.ray.numel(), device=DEV).split(CHUNK):
        v = _shade(sc, w, f.leaf[at], u[f.ray[at]], f.dn[f.ray[at]])
        dz = f.w[at][:, None] * g[f.ray[at]] * v.col * (1.0 - v.col)
        dg = (dz * v.dz).sum(1) * math.pi * v.sg * (1.0 - v.sg)
        row = torch.cat([dsig[at][:, None] * v.a, dg[:, None] * v.b, (dz[:, :, None] * v.H[:, None]).flatten(1)], 1)
        grad.index_add_(0, f.leaf[at], row)
    touched = torch.zeros(w.shape[0], dtype=torch.bool, device=DEV)
    touched[f.leaf[f.sig > 0]] = True
    return grad, touched


def _image_loss(rgb, target, rop, lam):
    """Value and gradient of the squared forward differences of |target - rgb|."""
    x = rgb.detach().clone().requires_grad_()
    total = 0.0
    for view in rop:
        E = (target[view.long()] - x[view.long()]).abs()
        total = total + lam * ((E[:, 1:] - E[:, :-1]).square().sum() + (E[1:] - E[:-1]).square().sum())
    total.backward()
    return float(total), x.grad


def _stored(sc, w, dtype):
    """The coefficients as the storage holds them."""
    if dtype != "fp8":
        return w if dtype == "f32" else w.bfloat16().float()
    K, out = sc.K, torch.empty_like(w)
    for lo, hi in ((0, K), (K, 2 * K), (2 * K, w.shape[1])):
        x = w[:, lo:hi].double()
        top = x.abs().amax(1, keepdim=True).clamp_min(1e-300)
        e = torch.exp2(torch.ceil(torch.log2(top / 448.0)))
        out[:, lo:hi] = ((x / e).float().to(torch.float8_e4m3fn).double() * e).float()
    return out


def exact(case, seed):
    with torch.no_grad():
        return _exact(case, seed)


def _exact(c, seed):
    sc, s = _scene_of(c), _inputs(c, seed)
    o, d = s.o.double().t().contiguous(), s.d.double().t().contiguous()
    u = s.t.double() * (sc.T - 1)
    w = _stored(sc, s.w if c["kind"] == "autograd" else sc.w, c["dtype"])
    if c["kind"] == "compose":
        return _exact_compose(c, sc, s, w, o, d)
    if c["kind"] == "autograd":
        f = _render(sc, w, o, d, u)
        grad, _ = _adjoint(sc, w, f, u, s.g_rgb.double(), s.g_alpha.double())
        return {"rgb": f.rgb, "alpha": f.alpha, "depth": f.depth, "grad": _padded(grad, (w.shape[1] + 3) // 4 * 4)}
    if c["kind"] in ("train", "batch"):
        f = _render(sc, w, o, d, u)
        r = f.rgb - s.target.double()
        loss, g = float(r.square().sum()) / s.n, 2.0 / s.n * r
        if c["kind"] == "train":
            with torch.enable_grad():
                more, extra = _image_loss(f.rgb, s.target.double(), s.ray_of_pixel, LAMBDA / s.n)
            loss, g = loss + more, g + extra
        grad, touched = _adjoint(sc, w, f, u, g, None)
        on, m0, v0, w0 = touched[:, None], s.m.double(), s.v.double(), sc.w.double()
        m = torch.where(on, BETA1 * m0 + (1 - BETA1) * grad, m0)
        v = torch.where(on, BETA2 * v0 + (1 - BETA2) * grad.square(), v0)
        step = LR * (m / (1 - BETA1 ** STEP)) / ((v / (1 - BETA2 ** STEP)).sqrt() + EPS)
        pad = (sc.w.shape[1] + 3) // 4 * 4
        return {"rgb": f.rgb, "alpha": f.alpha, "depth": f.depth, "tau": f.tau, "nseg": None,
                "loss": torch.tensor([loss], dtype=torch.float64), "m": _padded(m, pad), "v": _padded(v, pad),
                "master": _padded(torch.where(on, w0 - step, w0), pad), "storage": None}
    if c["kind"] == "slice":
        t = torch.full((sc.n,), float(s.times[0]), dtype=torch.float64, device=DEV) * (sc.T - 1)
        ny, rows = (sc.degree + 1) ** 2, []
        for at in torch.arange(sc.n, device=DEV).split(CHUNK):
            r, (a, b) = w[at].double(), _rows(sc, t[at])
            R, _, col, lm = _radial(sc.degree, math.pi * torch.sigmoid((b * r[:, sc.K:2 * sc.K]).sum(1)))
            part = r[:, 2 * sc.K:].view(-1, 3, sc.nh) * R[:, None, col]
            sh = torch.zeros(at.numel(), 3, ny, dtype=torch.float64, device=DEV)
            sh.index_add_(2, torch.tensor(lm, device=DEV), part)
            row = torch.zeros(at.numel(), (4 + 3 * ny + 3) // 4 * 4, dtype=torch.float64, device=DEV)
            row[:, 0] = (a * r[:, :sc.K]).sum(1).clamp_min(0.0)
            row[:, 4:4 + 3 * ny] = sh.flatten(1)
            rows.append(row)
        f = _render(sc, w, o, d, u)
        return {"rgb": f.rgb, "alpha": f.alpha, "depth": f.depth, "tau": f.tau, "nseg": None,
                "slice": torch.cat(rows)}
    edits = leaf = None
    if c["kind"] == "edit":
        f = _render(sc, w, o, d, u)
        gone = -torch.expm1(-f.before - f.sd) >= 0.99
        last = torch.full((s.n,), f.ray.numel(), dtype=torch.int64, device=DEV)
        at = torch.nonzero(gone).reshape(-1)
        last.scatter_reduce_(0, f.ray[at], at, "amin")
        hit = torch.nonzero(last < f.ray.numel()).reshape(-1)
        leaf = f.leaf[last[hit]]
        acc = torch.zeros(sc.n, 4, dtype=torch.float64, device=DEV)
        acc.index_add_(0, leaf, torch.cat([s.color[hit].double(), torch.ones(hit.numel(), 1, device=DEV).double()], 1))
        edits = torch.zeros(sc.n, 8, dtype=torch.float64, device=DEV)
        edits[:, 3], edits[:, 4] = -1.0, 2.0
        on = acc[:, 3] > 0
        edits[on, :3], edits[on, 4] = acc[on, :3] / acc[on, 3:], 0.0
    f = _render(sc, w, o, d, u, edit=edits)
    out = {"rgb": f.rgb, "alpha": f.alpha, "depth": f.depth, "tau": f.tau, "nseg": None}
    if c["kind"] == "edit":
        out.update(leaf=None, edits=edits)
    elif c["kind"] == "lit":
        lf = _render(sc, w, s.lo.double().t().contiguous(), s.ld.double().t().contiguous(),
                     s.lt.double() * (sc.T - 1))
        out["shadow"] = _blur(lf.alpha[s.light_map.reshape(-1).long()].view(LIGHT, LIGHT))[None]
        out["lit"] = _spotlight(s, o, f, out["shadow"][0])
    return out


def _blur(img):
    r = int(3 * BLUR + 0.5)
    k = torch.exp(-torch.arange(-r, r + 1, dtype=torch.float64, device=DEV).square() / (2 * BLUR * BLUR))
    k = k / k.sum()
    x = torch.nn.functional.pad(img[None, None], (r, r, r, r), mode="replicate")
    x = torch.nn.functional.conv2d(x, k.view(1, 1, 1, -1))
    return torch.nn.functional.conv2d(x, k.view(1, 1, -1, 1))[0, 0]


def _spotlight(s, o, f, shadow):
    eye, fwd, right, up = (torch.as_tensor(np.asarray(v), device=DEV)
                           for v in (s.light.eye, s.light.forward, s.light.right, s.light.up))

    def fall(p):
        return R_REF ** 2 / (p - eye).square().sum(1)
    some = torch.isfinite(f.depth)
    X = o + torch.where(some, f.depth, 0.0)[:, None] * f.dn
    lit = torch.where(some[:, None], f.rgb * fall(X)[:, None], f.rgb)
    t = torch.where(f.dn[:, 2] != 0, (GROUND - o[:, 2]) / f.dn[:, 2], -1.0)
    on = torch.isfinite(t) & (t > 0)
    P = o + torch.where(on, t, 0.0)[:, None] * f.dn
    v = P - eye
    z, th = v @ fwd, math.tan(math.radians(s.light.fov_y_deg) / 2)
    px = ((v @ right) / z / th + 1.0) * LIGHT / 2 - 0.5
    py = (1.0 - (v @ up) / z / th) * LIGHT / 2 - 0.5
    x0, y0, al = px.floor(), py.floor(), torch.zeros_like(px)
    for dx in (0, 1):
        for dy in (0, 1):
            x, y = x0 + dx, y0 + dy
            ok = (z > 0) & (x >= 0) & (x < LIGHT) & (y >= 0) & (y < LIGHT)
            texel = shadow[torch.where(ok, y, 0.0).long(), torch.where(ok, x, 0.0).long()]
            weight = (1 - (px - x).abs()) * (1 - (py - y).abs())
            al = al + torch.where(ok, weight * texel, 0.0)
    ground = ((1 - f.alpha) * (1 - al) * fall(P))[:, None] * torch.tensor(ALBEDO, device=DEV).double()
    return torch.where(on[:, None], lit + ground, lit)


def _exact_compose(c, sc, s, w, o, d):
    layers, length = [], d.norm(dim=1)
    for p in s.prims:
        M = torch.as_tensor(p.transform.astype(np.float32), device=DEV).double()
        inv = torch.linalg.inv(M[:, :3])
        lo, ld = (o - M[:, 3]) @ inv.t(), d @ inv.t()
        u = torch.remainder(s.t.double() * (sc.T - 1) + float(np.float32(p.time_offset)), sc.T - 1)
        f = _render(sc, w, lo, ld, u, scale=length / ld.norm(dim=1))
        tint = torch.as_tensor(p.tint.astype(np.float32), device=DEV).double()
        layers.append((f.rgb * tint, f.alpha, f.depth))
    C, A, D = (torch.stack(x) for x in zip(*layers))
    if c["mode"] == "sorted":
        by = torch.argsort(D, dim=0, stable=True)
        C, A = C.gather(0, by[..., None].expand_as(C)), A.gather(0, by)
        rgb, alpha = torch.zeros_like(C[0]), torch.zeros_like(A[0])
        for j in range(C.shape[0]):
            rgb = rgb + (1 - alpha)[:, None] * C[j]
            alpha = alpha + (1 - alpha) * A[j]
        return {"rgb": rgb, "alpha": alpha, "depth": D.amin(0)}
    rgb, alpha, depth = C[0], A[0], D[0]
    for j in range(1, C.shape[0]):
        front = D[j] <= depth
        rgb = torch.where(front[:, None], (1 - A[j])[:, None] * rgb + C[j], rgb + (1 - alpha)[:, None] * C[j])
        alpha, depth = alpha + A[j] * (1 - alpha), torch.where(front, D[j], depth)
    return {"rgb": rgb, "alpha": alpha, "depth": depth}
