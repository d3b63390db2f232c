"""The work that users of this framework have it do, as cases that can be timed and checked.

Every case is one pass through public entry points (``paper_2403_16862_gb300.api`` and ``batch``) on inputs made
from a seed: octree scenes with log-normal leaf weights, hash-grid tables, pinhole views and N(0, 1) upstream
gradients.  ``listed()`` names the cases, ``draw(rng)`` gives others of the same ranges, ``exact(case, seed)``
evaluates the same outputs in 64 bits with plain torch.

In ``exact`` the decisions that the entry points document as FP32 (projected pixel, depth order, contracted
position) are taken in FP32, everything after them in FP64.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_2403_16862_gb300 import _binding as B
from paper_2403_16862_gb300 import api
from paper_2403_16862_gb300.batch import ViewBatch

DEV = "cuda:0"
T_MIN, ALPHA_MAX = 1e-4, 0.99


def listed():
    return [
        # The smallest call: a probe of the field at a few thousand positions (an octree refresh, a debug view).
        dict(name="query_4k", kind="query", n=4_099, log2_T=19, levels=16, bf16=False, train=False),
        # The grid as a trainable layer: forward and table gradient through autograd, an odd count.
        dict(name="query_train_1m", kind="query", n=1_000_003, log2_T=19, levels=16, bf16=False, train=True),
        # The grid in inference precision: BF16 table beyond L2, BF16 features, one 8M-sample cloud.
        dict(name="query_8m_bf16", kind="query", n=8_388_608, log2_T=21, levels=16, bf16=True, train=False),
        # The plain rasterizer on a small cloud with given opacities, forward and backward: launches count.
        dict(name="raster_64k", kind="raster", n=65_536, F=8, W=256, H=256, head=False, leaves=0),
        # The rasterizer as a layer of a training step (64 channels, opacity from channel 0), an odd image.
        dict(name="raster_train_1m", kind="raster", n=1_000_003, F=64, W=641, H=417, head=True, leaves=65_536),
        # Inference from a pre-extracted global cloud: 67M BF16 points, forward only.
        dict(name="render_67m_bf16", kind="render", n=67_108_864, W=1280, H=832, bf16=True, leaves=65_536),
        # One training view, sampling to table gradient, with the fused backward and kept buffers.
        dict(name="view_train_4m", kind="view", n=4_194_304, W=1280, H=832, log2_T=19, bf16=False, leaves=65_536),
        # The largest training view: BF16 storage, a 2^21 table, a million leaves, full HD.
        dict(name="view_train_16m_bf16", kind="view", n=16_777_216, W=1920, H=1080, log2_T=21, bf16=True,
             leaves=1_048_576),
        # A batch of small training views as one graph with the persistent front end.
        dict(name="batch_16x256k", kind="batch", views=16, n=262_144, W=320, H=240, log2_T=19, bf16=False,
             leaves=65_536),
        # The view-dependent (spherical harmonics) variant, forward and backward.
        dict(name="view_sh_500k", kind="sh", n=500_009, W=637, H=411, log2_T=19, leaves=65_536),
        # The octree's share of a training step: per-point blending weights and the probability updates (its
        # subdivision and pruning run once in hundreds of steps).
        dict(name="octree_1m", kind="octree", n=1_048_576, W=640, H=416, leaves=65_536),
        # Inference with view-specific sampling and four-fold multisampling.
        dict(name="multisample_4x1m", kind="multisample", n=1_048_576, k=4, W=1237, H=822, log2_T=19, leaves=262_144),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def image(lo, hi):
        h = log_int(lo, hi)
        return int(h * rng.uniform(1.0, 1.8)), h

    kind = rng.choice(["query", "query", "raster", "raster", "render", "view", "view", "batch", "sh", "octree",
                       "multisample"])
    if kind == "query":
        train = rng.random() < 0.5
        return dict(kind=kind, n=log_int(1_000, 4_000_000 if train else 16_000_000), log2_T=rng.randint(14, 21),
                    levels=rng.choice([8, 16, 16, 16]), bf16=(not train) and rng.random() < 0.5, train=train)
    if kind == "raster":
        W, H = image(48, 700)
        F = rng.choice([3, 4, 8, 12, 32, 64, 64, 128])
        n = log_int(2_000, 1_500_000)
        return dict(kind=kind, n=n, F=F, W=W, H=H, head=F >= 4 and rng.random() < 0.5,
                    leaves=rng.choice([0, log_int(5_000, 65_536)]))
    if kind == "render":
        W, H = image(240, 1080)
        return dict(kind=kind, n=log_int(200_000, 40_000_000), W=W, H=H, bf16=rng.random() < 0.7,
                    leaves=log_int(20_000, 500_000))
    if kind == "view":
        W, H = image(96, 1080)
        return dict(kind=kind, n=log_int(20_000, 8_000_000), W=W, H=H, log2_T=rng.randint(16, 21),
                    bf16=rng.random() < 0.4, leaves=log_int(5_000, 300_000))
    if kind == "batch":
        W, H = image(96, 480)
        return dict(kind=kind, views=rng.randint(2, 16), n=log_int(20_000, 500_000), W=W, H=H,
                    log2_T=rng.randint(16, 20), bf16=rng.random() < 0.5, leaves=log_int(5_000, 100_000))
    if kind == "sh":
        W, H = image(96, 800)
        return dict(kind=kind, n=log_int(10_000, 2_000_000), W=W, H=H, log2_T=rng.randint(16, 20),
                    leaves=log_int(5_000, 100_000))
    if kind == "octree":
        W, H = image(96, 832)
        return dict(kind=kind, n=log_int(20_000, 4_000_000), W=W, H=H, leaves=log_int(5_000, 300_000))
    W, H = image(120, 900)
    return dict(kind="multisample", n=log_int(20_000, 2_000_000), k=rng.randint(1, 4), W=W, H=H,
                log2_T=rng.randint(16, 20), leaves=log_int(5_000, 300_000))


# ------------------------------------------------------------------ inputs ---
def resolutions(levels):
    """Geometric from 16 to 4096."""
    b = 256.0 ** (1.0 / (levels - 1))
    return [int(math.floor(16 * b ** l + 1e-9)) for l in range(levels)]


def layout(res, log2_T):
    """(first row of every level, dense flags, rows in all): levels start on multiples of 16 rows."""
    T, off, start, dense = 1 << log2_T, 0, [], []
    for r in res:
        d = (r + 1) ** 3 <= T
        off = (off + 15) // 16 * 16
        start.append(off)
        dense.append(d)
        off += (r + 1) ** 3 if d else T
    return start, dense, (off + 15) // 16 * 16


def generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 17)
    return g


def make_octree(n_leaves, g):
    """(centers f32 [L,3], levels i32 [L], weights f64 [L]) in the unit cube: a uniform start grid, random
    refinement, pruning to exactly n_leaves, Morton order, log-normal(0, 1.5) weights that sum to one."""
    start = 4 if n_leaves < 400_000 else 6
    side = 1 << start
    ijk = torch.cartesian_prod(*[torch.arange(side, device=DEV)] * 3)
    lv = torch.full((side ** 3,), start, dtype=torch.int64, device=DEV)
    while lv.numel() < n_leaves:
        k = max(1, (n_leaves - lv.numel()) // 24)
        perm = torch.randperm(lv.numel(), generator=g, device=DEV)
        perm = perm[lv[perm] < 12]
        split, keep = perm[:k], torch.ones(lv.numel(), dtype=torch.bool, device=DEV)
        keep[split] = False
        child = torch.cartesian_prod(*[torch.arange(2, device=DEV)] * 3)
        kids = (2 * ijk[split][:, None] + child[None]).reshape(-1, 3)
        ijk = torch.cat([ijk[keep], kids])
        lv = torch.cat([lv[keep], (lv[split] + 1).repeat_interleave(8)])
    pick = torch.randperm(lv.numel(), generator=g, device=DEV)[:n_leaves]
    ijk, lv = ijk[pick], lv[pick]
    code, at = torch.zeros_like(lv), ijk << (12 - lv)[:, None]
    for b in range(12):
        for a in range(3):
            code |= ((at[:, a] >> b) & 1) << (3 * b + a)
    order = torch.argsort(code)
    ijk, lv = ijk[order], lv[order]
    centers = ((ijk.double() + 0.5) * torch.exp2(-lv.double())[:, None]).float().contiguous()
    w = torch.exp(1.5 * torch.randn(n_leaves, dtype=torch.float64, generator=g, device=DEV))
    return centers, lv.to(torch.int32), w / w.sum()


def leaf_points(tree, n, g):
    """(leaf i32 [n], pos f32 [n,3]): n samples grouped by leaf, uniform in their leaves."""
    c, l, w = tree
    cdf = torch.cumsum(w, 0)
    u = torch.rand(n, dtype=torch.float64, generator=g, device=DEV) * cdf[-1]
    leaf = torch.searchsorted(cdf, u).clamp_(max=l.numel() - 1)
    del u
    leaf = torch.sort(leaf)[0]
    pos = torch.empty(n, 3, dtype=torch.float32, device=DEV)
    for a in range(0, n, 1 << 23):
        s = leaf[a:a + (1 << 23)]
        r = torch.rand(s.numel(), 3, generator=g, device=DEV)
        pos[a:a + s.numel()] = c[s] + (r - 0.5) * torch.exp2(-l[s].float())[:, None]
    return leaf.to(torch.int32), pos


def make_table(rows, bf16, g):
    t = torch.randn(rows, 4, generator=g, device=DEV) * 0.1
    t += (torch.rand(rows, 4, generator=g, device=DEV) * 2 - 1) * 1e-4
    return t.bfloat16() if bf16 else t


def normal(shape, g):
    return torch.randn(shape, generator=g, device=DEV)


def point_features(n, F, bf16, g):
    """Rows as the grid query gives them: small values around zero."""
    f = torch.empty(n, F, dtype=torch.bfloat16 if bf16 else torch.float32, device=DEV)
    for a in range(0, n, 1 << 22):
        f[a:a + (1 << 22)] = torch.randn(min(1 << 22, n - a), F, generator=g, device=DEV) * 0.05
    return f


def front_camera(W, H):
    """In front of the unit cube, looking down +z; the focal length follows the image height."""
    f = 900.0 * H / 832.0
    return types.SimpleNamespace(R=np.eye(3, dtype=np.float32), t=np.array([-0.5, -0.5, 1.2], np.float32), fx=f, fy=f,
                                 cx=W / 2.0, cy=H / 2.0, width=W, height=H, near=0.01, far=100.0)


def orbit_camera(W, H, k, n):
    """View k of n on a horizontal orbit around the cube's center."""
    a = 2.0 * math.pi * k / n
    c = np.full(3, 0.5)
    eye = c + 1.7 * np.array([math.sin(a), -0.25, -math.cos(a)])
    z = (c - eye) / np.linalg.norm(c - eye)
    x = np.cross([0.0, 1.0, 0.0], z)
    x /= np.linalg.norm(x)
    R = np.stack([x, np.cross(z, x), z])
    f = 900.0 * H / 832.0
    return types.SimpleNamespace(R=R.astype(np.float32), t=(-R @ eye).astype(np.float32), fx=f, fy=f, cx=W / 2.0,
                                 cy=H / 2.0, width=W, height=H, near=0.01, far=100.0)


def make_inputs(c, seed):
    """The case's arrays, made from the seed alone."""
    g = generator(seed)
    i = types.SimpleNamespace(seed=int(seed))
    kind = c["kind"]
    if kind in ("query", "view", "batch", "sh", "multisample"):
        i.res = resolutions(c.get("levels", 16))
        i.start, i.dense, i.rows = layout(i.res, c["log2_T"])
        i.table = make_table(i.rows, c.get("bf16", False), g)
    if c.get("leaves"):
        i.tree = make_octree(c["leaves"], g)
    if kind == "query":
        # positions as the sampler gives them: in a few thousand leaves, grouped by leaf
        i.pos = leaf_points(make_octree(16_384, g), c["n"], g)[1]
        if c["train"]:
            i.dh = normal((c["n"], 4 * c["levels"]), g)
    elif kind == "raster":
        i.cam = front_camera(c["W"], c["H"])
        if c["leaves"]:
            i.pos = leaf_points(i.tree, c["n"], g)[1]
        else:
            i.pos = torch.rand(c["n"], 3, generator=g, device=DEV)
        if c["head"]:
            i.feat, i.opacity = point_features(c["n"], c["F"], False, g), None
        else:
            i.feat = normal((c["n"], c["F"]), g)
            i.opacity = 0.05 + 0.9 * torch.rand(c["n"], generator=g, device=DEV)
        i.d_image = normal((c["H"], c["W"], c["F"]), g)
    elif kind == "render":
        i.cam = front_camera(c["W"], c["H"])
        i.pos = leaf_points(i.tree, c["n"], g)[1]
        i.feat = point_features(c["n"], 64, c["bf16"], g)
    elif kind == "view":
        i.cam = front_camera(c["W"], c["H"])
        i.d_image = normal((c["H"], c["W"], 64), g)
    elif kind == "batch":
        i.cams = [orbit_camera(c["W"], c["H"], k, c["views"]) for k in range(c["views"])]
        i.d_images = [normal((c["H"], c["W"], 64), g) for _ in i.cams]
    elif kind == "sh":
        # a scene that reaches beyond the unit ball of its normalisation, where the contraction bends
        i.cam = orbit_camera(c["W"], c["H"], 1, 7)
        i.center, i.radius = (0.5, 0.5, 0.5), 0.4
        i.pos = leaf_points(i.tree, c["n"], g)[1]
        i.d_image = normal((c["H"], c["W"], 4), g)
    elif kind == "octree":
        i.cam = front_camera(c["W"], c["H"])
        i.leaf, i.pos = leaf_points(i.tree, c["n"], g)
        i.feat = point_features(c["n"], 64, False, g)
        L = c["leaves"]
        i.p = torch.rand(L, dtype=torch.float64, generator=g, device=DEV).square_()
        i.q = 0.55 * torch.rand(L, dtype=torch.float64, generator=g, device=DEV)
    elif kind == "multisample":
        i.cam = orbit_camera(c["W"], c["H"], 2, 9)
        i.cam.fx = i.cam.fy = 1.6 * i.cam.fx  # a close view: part of the scene lies outside it
    return i


def grid_desc(c, i):
    dt = torch.bfloat16 if c.get("bf16") else torch.float32
    return api.hashgrid_desc(i.res, c["log2_T"], table_dtype=dt, out_dtype=dt)


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    s = make_inputs(c, seed)
    s.kind, s.c = kind, c
    if hasattr(s, "res"):
        s.desc = grid_desc(c, s)
    if kind == "query" and c["train"]:
        s.table.requires_grad_(True)
    elif kind == "raster":
        s.opts = api.RasterOptions(n_channels=c["F"], head_mode=c["head"])
        s.feat.requires_grad_(True)
        if s.opacity is not None:
            s.opacity.requires_grad_(True)
    elif kind == "render":
        # a viewer keeps its workspace and its frame buffers
        s.opts = api.RasterOptions(n_channels=64, head_mode=True, bf16=c["bf16"])
        s.ws = api.workspace(api.rasterize_workspace_size(s.cam, s.opts, c["n"]), DEV)
        s.out = frame_buffers(c, 64, s.opts.dtype)
    elif kind == "view":
        # a training loop keeps its buffers
        n = c["n"]
        s.opts = api.RasterOptions(n_channels=64, head_mode=True, bf16=c["bf16"])
        s.ws_s = api.workspace(B.inpc_sample_workspace_size(c["leaves"], n), DEV)
        s.sample = (torch.empty(n, dtype=torch.int32, device=DEV), torch.empty(n, 3, device=DEV))
        s.h = torch.empty(n, 64, dtype=s.opts.dtype, device=DEV)
        s.ws = api.workspace(api.rasterize_bwd_hashgrid_workspace_size(s.cam, s.opts, s.desc, n), DEV)
        s.out = frame_buffers(c, 64, s.opts.dtype)
        s.grad = torch.zeros(s.rows, 4, device=DEV)
    elif kind == "batch":
        s.batch = ViewBatch(*s.tree, 1.0, s.desc, s.table, s.cams, c["n"], s.d_images, seed=s.seed, n_streams=4,
                            bf16=c["bf16"], tune=False, persistent=True).capture()
    elif kind == "sh":
        s.grad = torch.zeros(s.rows, 4, device=DEV)
    elif kind == "octree":
        # the forward of the same step has filled the workspace
        s.opts = api.RasterOptions(n_channels=64, head_mode=True)
        _, _, s.n_contrib, s.ws = api.rasterize_fwd(s.cam, s.opts, s.pos, s.feat)
    return s


def frame_buffers(c, F, dtype):
    return (torch.empty(c["H"], c["W"], F, dtype=dtype, device=DEV), torch.empty(c["H"], c["W"], device=DEV),
            torch.empty(c["H"], c["W"], dtype=torch.int32, device=DEV))


def run(s):
    kind, c = s.kind, s.c
    if kind == "query":
        if not c["train"]:
            return {"h": api.query_hashgrid(s.desc, s.table, s.pos)}
        h = api.HashGridQuery.apply(s.table, s.pos, s.desc)
        (grad,) = torch.autograd.grad(h, s.table, s.dh)
        return {"h": h.detach(), "grad": grad}
    if kind == "raster":
        img, T, nc = api.Rasterize.apply(s.pos, s.feat, s.opacity, s.cam, s.opts)
        leaves = [s.feat] if s.opacity is None else [s.feat, s.opacity]
        return {"image": img.detach(), "T": T, "n": nc, "grads": torch.autograd.grad(img, leaves, s.d_image)}
    if kind == "render":
        img, T, nc, _ = api.rasterize_fwd(s.cam, s.opts, s.pos, s.feat, ws=s.ws, out=s.out)
        return {"image": img, "T": T, "n": nc}
    if kind == "view":
        leaf, pos = api.sample_octree(*s.tree, 1.0, s.seed, 3, c["n"], ws=s.ws_s, out=s.sample)
        h = api.query_hashgrid(s.desc, s.table, pos, out=s.h)
        img, T, nc, _ = api.rasterize_fwd(s.cam, s.opts, pos, h, ws=s.ws, out=s.out)
        s.grad.zero_()
        api.rasterize_bwd_hashgrid(s.cam, s.opts, s.desc, pos, h, T, nc, s.d_image, s.ws, s.grad)
        return {"leaf": leaf, "pos": pos, "image": img, "T": T, "n": nc, "grad": s.grad}
    if kind == "batch":
        s.batch.step()
        return {"views": [[v["img"], v["T"], v["nc"]] for v in s.batch.views], "grad": s.batch.grad_table}
    if kind == "sh":
        s.grad.zero_()
        img, T, nc = api.render_view_sh(s.pos, s.desc, s.table, s.cam, s.center, s.radius, s.d_image, s.grad)
        return {"image": img, "T": T, "n": nc, "grad": s.grad}
    if kind == "octree":
        b = api.point_weights(s.cam, s.opts, s.pos, s.n_contrib, s.ws)
        p, q = api.octree_update(s.leaf, b, s.p, s.q)
        return {"b": b, "p": p, "q": q}
    return {"image": api.multisample_render(s.tree, 1.0, s.desc, s.table, s.cam, s.seed, c["n"], k=c["k"])}


def work(case):
    """Every input read once and every output written once; multiply-adds as two operations."""
    c = case
    n, kind = c["n"], c["kind"]
    e = 2 if c.get("bf16") else 4
    pix = c.get("W", 0) * c.get("H", 0)
    levels = c.get("levels", 16)
    rows = layout(resolutions(levels), c["log2_T"])[2] if "log2_T" in c else 0
    # a few points touch a few rows
    rows = min(rows, c.get("views", 1) * c.get("k", 1) * n * levels * 8)
    corner = n * levels * 8 * 11  # weight and four multiply-adds per corner
    leaves = 24 * c.get("leaves", 0)
    if kind == "query":
        by, fl = 12 * n + 4 * e * rows + 4 * levels * e * n, corner
        if c["train"]:
            by, fl = by + 16 * levels * n + 16 * rows, 2 * fl
    elif kind == "raster":
        F = c["F"]
        by = (12 + 4 * F) * n + (4 * F + 8) * pix + 4 * F * pix + 4 * F * n + (0 if c["head"] else 8 * n)
        fl = 60 * n + 4 * n * F * 8
    elif kind == "render":
        by, fl = (12 + 64 * e) * n + (64 * e + 8) * pix, 60 * n + 64 * 2 * 30 * pix
    elif kind == "view":
        by = leaves + 16 * n + 4 * e * rows + 16 * rows + (64 * e + 8) * pix + 256 * pix
        fl = 2 * corner + 250 * n + 64 * 4 * 30 * pix
    elif kind == "batch":
        v = c["views"]
        by = leaves + 4 * e * rows + 16 * rows + v * ((64 * e + 8) * pix + 256 * pix)
        fl = v * (2 * corner + 250 * n + 64 * 4 * 30 * pix)
    elif kind == "sh":
        by, fl = 12 * n + 32 * rows + (16 + 8 + 16) * pix, 2 * corner + 500 * n
    elif kind == "octree":
        by, fl = 12 * n + 4 * n + 4 * n + 4 * pix + 32 * c["leaves"], 60 * n
    else:
        by = leaves + 16 * rows + 256 * pix
        fl = c["k"] * (corner + 250 * n + 64 * 2 * 30 * pix)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------ 64-bit values ---
def f32(x):
    return x.to(torch.float32)


def exact_cells(pos, N):
    x = pos.clamp(0.0, 1.0).double() * N
    cell = torch.floor(x).clamp_(max=N - 1)
    return cell.to(torch.int64), x - cell


def exact_corners(i, log2_T, pos):
    """Per level and corner: (level, row, weight) of every point."""
    for l, N in enumerate(i.res):
        cell, f = exact_cells(pos, N)
        for k in range(8):
            v = [cell[:, a] + ((k >> a) & 1) for a in range(3)]
            w = [f[:, a] if (k >> a) & 1 else 1.0 - f[:, a] for a in range(3)]
            if i.dense[l]:
                row = v[0] + (N + 1) * (v[1] + (N + 1) * v[2])
            else:
                m = (1 << log2_T) - 1
                row = (v[0] ^ ((v[1] * 2654435761) & m) ^ ((v[2] * 805459861) & m)) & m
            yield l, row + i.start[l], w[0] * w[1] * w[2]


def exact_query(i, log2_T, pos):
    h = torch.zeros(pos.shape[0], len(i.res), 4, dtype=torch.float64, device=DEV)
    table = i.table.detach()
    for a in range(0, pos.shape[0], 1 << 21):
        for l, row, w in exact_corners(i, log2_T, pos[a:a + (1 << 21)]):
            h[a:a + (1 << 21), l] += w[:, None] * table[row].double()
    return h.reshape(pos.shape[0], -1)


def exact_adjoint(i, log2_T, pos, dh, grad=None):
    grad = torch.zeros(i.rows, 4, dtype=torch.float64, device=DEV) if grad is None else grad
    dh = dh.reshape(pos.shape[0], len(i.res), 4)
    for a in range(0, pos.shape[0], 1 << 21):
        for l, row, w in exact_corners(i, log2_T, pos[a:a + (1 << 21)]):
            grad.index_add_(0, row, w[:, None] * dh[a:a + (1 << 21), l].double())
    return grad


def fma32(a, b, c):
    return f32(float(a) * b.double() + c.double())


def exact_project(cam, pos):
    """(u, v, depth, kept): the projection in FP32, each step rounded once."""
    x, y, z = pos[:, 0], pos[:, 1], pos[:, 2]
    R = np.asarray(cam.R, np.float32)
    t = torch.tensor(np.asarray(cam.t, np.float32), device=DEV)
    p = [fma32(R[k, 2], z, fma32(R[k, 1], y, fma32(R[k, 0], x, t[k]))) for k in range(3)]
    near, far = np.float32(cam.near), np.float32(cam.far)
    keep = (p[2] > float(near)) & (p[2] < float(far))
    u = fma32(np.float32(cam.fx), p[0] / p[2], torch.tensor(np.float32(cam.cx), device=DEV))
    v = fma32(np.float32(cam.fy), p[1] / p[2], torch.tensor(np.float32(cam.cy), device=DEV))
    return u, v, p[2], keep


class ExactRaster:
    """Forward (and backward) of the bilinear splatting in FP64: fragments ordered by (pixel, depth, point)."""

    def __init__(self, cam, pos, alpha_h, feat, F, head):
        self.W, self.H, self.F, self.head, self.feat, self.n = cam.width, cam.height, F, head, feat, pos.shape[0]
        P = self.P = self.W * self.H
        u, v, d, keep = exact_project(cam, pos)
        keep &= (u >= -0.5) & (u < self.W + 0.5) & (v >= -0.5) & (v < self.H + 0.5)
        ids = torch.nonzero(keep)[:, 0]
        ids = ids[torch.argsort(d[ids], stable=True)]
        su, sv = (u[ids].double() - 0.5), (v[ids].double() - 0.5)
        i0, j0 = torch.floor(f32(su)).long(), torch.floor(f32(sv)).long()
        fu, fv = su - i0, sv - j0
        pix = []
        for k in range(4):
            px, py = i0 + (k & 1), j0 + (k >> 1)
            inside = (px >= 0) & (px < self.W) & (py >= 0) & (py < self.H)
            pix.append(torch.where(inside, py * self.W + px, P).to(torch.int32))
        pix = torch.stack(pix, 1).reshape(-1)
        pix, order = torch.sort(pix, stable=True)
        self.start = torch.searchsorted(pix, torch.arange(P + 1, device=DEV, dtype=torch.int32))
        total = int(self.start[P])
        # whole pixels at a time: about 2^24 fragments each
        self.parts = []
        self.T = torch.ones(P, dtype=torch.float64, device=DEV)
        a = 0
        starts = self.start.cpu().numpy()
        while a < P:
            b = int(np.searchsorted(starts, starts[a] + (1 << 24), side="right")) - 1
            b = min(P, max(a + 1, b))
            lo, hi = int(starts[a]), int(starts[b])
            if hi > lo:
                o, q = order[lo:hi], pix[lo:hi].long()
                r, k = o >> 2, o & 3
                w = torch.where((k & 1) == 1, fu[r], 1 - fu[r]) * torch.where(k >= 2, fv[r], 1 - fv[r])
                al = alpha_h[ids[r]] * w
                free = al <= ALPHA_MAX
                al = al.clamp(max=ALPHA_MAX)
                lg = torch.log1p(-al)
                cum = torch.cumsum(lg, 0)
                first = (self.start[q] - lo).long()
                before = cum - lg - (cum[first] - lg[first])
                blended = before >= math.log(T_MIN)
                sel = torch.nonzero(blended)[:, 0]
                last = torch.zeros(P, dtype=torch.float64, device=DEV)
                last.index_add_(0, q[sel], lg[sel])
                self.T[a:b] = torch.exp(last[a:b])
                self.parts.append((ids[r[sel]], q[sel], al[sel], torch.exp(before[sel]), w[sel], free[sel]))
            a = b
        assert total == starts[P]

    def colors(self, id_):
        c = self.feat[id_].double()
        if self.head:
            c[:, 0] = 1.0
        return c

    def image(self):
        img = torch.zeros(self.P, self.F, dtype=torch.float64, device=DEV)
        for id_, q, al, T, _, _ in self.parts:
            for a in range(0, id_.numel(), 1 << 21):
                s = slice(a, a + (1 << 21))
                img.index_add_(0, q[s], (T[s] * al[s])[:, None] * self.colors(id_[s]))
        return img.reshape(self.H, self.W, self.F)

    def final_T(self):
        return self.T.reshape(self.H, self.W)

    def weights(self):
        b = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        for id_, _, al, T, w, _ in self.parts:
            b.index_add_(0, id_, w * T * al)
        return b

    def backward(self, d_image):
        """(d feat [n,F] with channel 0 empty in head mode, d alpha_h [n])"""
        g = d_image.reshape(self.P, self.F).double()
        df = torch.zeros(self.n, self.F, dtype=torch.float64, device=DEV)
        da = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        for id_, q, al, T, w, free in self.parts:
            dot = torch.empty_like(al)
            for a in range(0, id_.numel(), 1 << 21):
                s = slice(a, a + (1 << 21))
                gq = g[q[s]]
                dot[s] = (self.colors(id_[s]) * gq).sum(1)
                df.index_add_(0, id_[s], (T[s] * al[s])[:, None] * gq)
            term = T * al * dot
            tot = torch.zeros(self.P, dtype=torch.float64, device=DEV).index_add_(0, q, term)
            cum = torch.cumsum(term, 0)
            first = torch.searchsorted(q, q)
            behind = tot[q] - (cum - (cum[first] - term[first]))
            da.index_add_(0, id_, torch.where(free, w * (T * dot - behind / (1 - al)), 0.0))
        if self.head:
            df[:, 0] = 0.0
        return df, da


def alpha_of(h0):
    return -torch.expm1(-torch.exp(h0.double()))


def head_gradient(df, da, h0):
    """The opacity path into channel 0 (head mode)."""
    e = torch.exp(h0.double())
    df[:, 0] = da * e * torch.exp(-e)
    return df


def philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    M = 0xFFFFFFFF
    k0, k1 = seed & M, (seed >> 32) & M

    def mul(a, m):  # 32 x 32 -> (high, low) without overflowing 63 bits
        lo, hi = a * (m & 0xFFFF), a * (m >> 16)
        t = hi + (lo >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        ha, la = mul(c0, 0xD2511F53)
        hb, lb = mul(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = hb ^ c1 ^ k0, lb, ha ^ c3 ^ k1, la
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c0, c1, c2, c3


def exact_cdf(w):
    return torch.cumsum(torch.round(w / w.max() * 2.0 ** 29).long(), 0)


def words(slots, view, purpose, seed):
    z = torch.zeros_like(slots)
    return philox(slots & 0xFFFFFFFF, slots >> 32, z + view, z + purpose, seed)


def draw_leaves(cdf, slots, view, purpose, seed):
    """Smallest leaf whose cumulative weight exceeds floor(b Q / 2^53), b the draw's 53 random bits."""
    x, y, _, _ = words(slots, view, purpose, seed)
    Q = int(cdf[-1])
    bh, bl = ((y & 0x1FFFFF) << 6) | (x >> 26), x & 0x3FFFFFF  # 27 high, 26 low bits
    qh, ql = Q >> 26, Q & 0x3FFFFFF
    mid = bh * ql + ((bl * ql) >> 26) + bl * qh  # units of 2^26
    r = (bh * qh + (mid >> 26)) >> 1             # b Q >> 53
    return torch.searchsorted(cdf, r, right=True).clamp_(max=cdf.numel() - 1)


def draw_positions(tree, leaf, slots, view, purpose, seed):
    x, y, z, _ = words(slots, view, purpose, seed)
    u = torch.stack([x, y, z], 1) >> 8
    edge = torch.exp2(-tree[1][leaf].double())[:, None]
    return f32(tree[0][leaf].double() + (u.double() * 2.0 ** -24 - 0.5) * edge)


def exact_sample(tree, w, n, view, seed):
    """(leaf, pos): the sampler's list, grouped by leaf."""
    cdf = exact_cdf(w)
    counts = torch.zeros(cdf.numel(), dtype=torch.int64, device=DEV)
    for a in range(0, n, 1 << 23):
        s = torch.arange(a, min(n, a + (1 << 23)), device=DEV)
        counts += torch.bincount(draw_leaves(cdf, s, view, 0, seed), minlength=cdf.numel())
    leaf = torch.repeat_interleave(torch.arange(cdf.numel(), device=DEV), counts)
    pos = torch.empty(n, 3, device=DEV)
    for a in range(0, n, 1 << 23):
        s = torch.arange(a, min(n, a + (1 << 23)), device=DEV)
        pos[a:a + s.numel()] = draw_positions(tree, leaf[s], s, view, 1, seed)
    return leaf, pos


def exact_view_weights(tree, cam):
    """Leaf weight over (view depth x level factor), zero for leaves whose cube lies outside a frustum plane."""
    c, l, p = tree
    R, t = np.asarray(cam.R, np.float64), np.asarray(cam.t, np.float64)

    def to_cam(x):
        return [((R[k, 0] * x[0] + R[k, 1] * x[1]) + R[k, 2] * x[2]) + t[k] for k in range(3)]

    fx, fy, cx, cy = (float(np.float32(v)) for v in (cam.fx, cam.fy, cam.cx, cam.cy))
    near, far = float(np.float32(cam.near)), float(np.float32(cam.far))
    e = torch.exp2(-l.double())
    x0 = [c[:, a].double() for a in range(3)]
    out = [torch.ones_like(e, dtype=torch.bool) for _ in range(6)]
    for k in range(8):
        q = to_cam([x0[a] + (0.5 if (k >> a) & 1 else -0.5) * e for a in range(3)])
        tests = (q[2] <= near, q[2] >= far, fx * q[0] + cx * q[2] < 0, fx * q[0] + (cx - cam.width) * q[2] >= 0,
                 fy * q[1] + cy * q[2] < 0, fy * q[1] + (cy - cam.height) * q[2] >= 0)
        out = [o & s for o, s in zip(out, tests)]
    d = ((to_cam(x0)[2] - near).abs() / far).clamp(min=1e-8)
    w = p / (d * torch.exp2(0.5 * l.double()))
    return torch.where(torch.stack(out).any(0), 0.0, w)


def exact_sample_view(tree, w, cam, n, view, seed, rounds=8):
    leaf, pos = exact_sample(tree, w, n, view, seed)
    cdf = exact_cdf(w)
    for r in range(rounds):
        u, v, _, keep = exact_project(cam, pos)
        bad = torch.nonzero(~(keep & (u >= 0) & (u < cam.width) & (v >= 0) & (v < cam.height)))[:, 0]
        if not bad.numel():
            break
        leaf[bad] = draw_leaves(cdf, bad, view, 2 + 2 * r, seed)
        pos[bad] = draw_positions(tree, leaf[bad], bad, view, 3 + 2 * r, seed)
    return pos


def exact_view(i, log2_T, cam, pos, d_image, grad):
    h = exact_query(i, log2_T, pos)
    r = ExactRaster(cam, pos, alpha_of(h[:, 0]), h, 64, True)
    if d_image is not None:
        df, da = r.backward(d_image)
        exact_adjoint(i, log2_T, pos, head_gradient(df, da, h[:, 0]), grad)
    return r.image(), r.final_T()


def sh_basis(cam, pos):
    R, t = np.asarray(cam.R, np.float64), np.asarray(cam.t, np.float64)
    o = torch.tensor(-(R.T @ t), device=DEV)
    d = pos.double() - o
    x, y, z = (d / d.norm(dim=1, keepdim=True)).unbind(1)
    a, b, c = math.sqrt(1 / (4 * math.pi)), math.sqrt(3 / (4 * math.pi)), math.sqrt(15 / (4 * math.pi))
    return torch.stack([torch.full_like(x, a), b * y, b * z, b * x, c * x * y, c * y * z,
                        math.sqrt(5 / (16 * math.pi)) * (3 * z * z - 1), c * x * z,
                        math.sqrt(15 / (16 * math.pi)) * (x * x - y * y)], 1)


def exact_contract(pos, center, radius):
    """Into [0, 1]^3 in FP32, each step rounded once."""
    y = [(pos[:, a] - float(np.float32(center[a]))) / torch.tensor(radius, dtype=torch.float32, device=DEV) for a in range(3)]
    sq = f32(y[2].double() ** 2 + f32(y[1].double() ** 2 + f32(y[0].double() ** 2).double()).double())
    r = torch.sqrt(sq)
    sc = torch.where(r > 1, (2.0 - 1.0 / r) / r, torch.ones_like(r))
    return torch.stack([f32((a * sc).double() * 0.25 + 0.5) for a in y], 1)


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    i = make_inputs(c, seed)
    if kind == "query":
        out = {"h": exact_query(i, c["log2_T"], i.pos)}
        if c["train"]:
            out["grad"] = exact_adjoint(i, c["log2_T"], i.pos, i.dh)
        return out
    if kind == "raster":
        alpha = alpha_of(i.feat[:, 0]) if c["head"] else i.opacity.double()
        r = ExactRaster(i.cam, i.pos, alpha, i.feat, c["F"], c["head"])
        df, da = r.backward(i.d_image)
        grads = [head_gradient(df, da, i.feat[:, 0])] if c["head"] else [df, da]
        return {"image": r.image(), "T": r.final_T(), "n": None, "grads": grads}
    if kind == "render":
        r = ExactRaster(i.cam, i.pos, alpha_of(i.feat[:, 0]), i.feat, 64, True)
        return {"image": r.image(), "T": r.final_T(), "n": None}
    if kind == "view":
        grad = torch.zeros(i.rows, 4, dtype=torch.float64, device=DEV)
        leaf, pos = exact_sample(i.tree, i.tree[2], c["n"], 3, i.seed)
        img, T = exact_view(i, c["log2_T"], i.cam, pos, i.d_image, grad)
        return {"leaf": leaf.to(torch.int32), "pos": pos, "image": img, "T": T, "n": None, "grad": grad}
    if kind == "batch":
        grad = torch.zeros(i.rows, 4, dtype=torch.float64, device=DEV)
        views = []
        for v, cam in enumerate(i.cams):
            pos = exact_sample(i.tree, i.tree[2], c["n"], v, i.seed)[1]
            img, T = exact_view(i, c["log2_T"], cam, pos, i.d_images[v], grad)
            views.append([img, T, None])
        return {"views": views, "grad": grad}
    if kind == "sh":
        q = exact_contract(i.pos, i.center, i.radius)
        h = exact_query(i, c["log2_T"], q)
        Y = sh_basis(i.cam, i.pos)
        color = torch.einsum("nck,nk->nc", h[:, 1:37].reshape(-1, 4, 9), Y)
        r = ExactRaster(i.cam, i.pos, alpha_of(h[:, 0]), color, 4, False)
        dcol, da = r.backward(i.d_image)
        dh = torch.zeros_like(h)
        dh[:, 1:37] = (dcol[:, :, None] * Y[:, None, :]).reshape(-1, 36)
        dh = head_gradient(dh, da, h[:, 0])
        return {"image": r.image(), "T": r.final_T(), "n": None, "grad": exact_adjoint(i, c["log2_T"], q, dh)}
    if kind == "octree":
        b = ExactRaster(i.cam, i.pos, alpha_of(i.feat[:, 0]), i.feat, 64, True).weights()
        leaf, lam = i.leaf.long(), 0.9968
        mx = torch.full_like(i.p, -1.0).scatter_reduce_(0, leaf, b, "amax")
        mn = torch.full_like(i.p, 2.0).scatter_reduce_(0, leaf, b, "amin")
        p = torch.where(mx >= 0, torch.maximum(mx, lam * i.p), lam * i.p)
        q = torch.where(mx >= 0, torch.maximum(mx - mn, lam * i.q), lam * i.q)
        return {"b": b, "p": p, "q": q}
    w = exact_view_weights(i.tree, i.cam)
    acc = torch.zeros(c["H"], c["W"], 64, dtype=torch.float64, device=DEV)
    for v in range(c["k"]):
        pos = exact_sample_view(i.tree, w, i.cam, c["n"], v, i.seed)
        acc += exact_view(i, c["log2_T"], i.cam, pos, None, None)[0] / c["k"]
    return {"image": acc}
