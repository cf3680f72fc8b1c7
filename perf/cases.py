"""The workloads by which the speed of this library is judged.

Each case is one thing that a user of the library has it do, through the public entry points of
``paper_2404_11852_gb300.cicero`` (the binding of include/cicero.h) or ``.autograd``:

  frame   one full frame (cicero_render): the smallest preview, an ordinary odd-sized one, the
          800x800 frame of the benchmark with the BF16 MLP and with the plain FP32 one, and the
          FP32-class split-BF16 MLP
  grad    cicero_render_backward for a ragged set of rays (grid gradients only, FP16 grid)
  train   a whole training step's forward and backward through autograd (grid and MLP gradients)
  rays    cicero_render_rays: the forward of explicit rays alone
  window  the benchmark's SpaRW window: reference frame, 16 warps in one batch, their holes
  path    SpaRW over a trajectory (the cicero_pipeline handle, reference on a second stream)
  warp    one warp to a new view with the warp-angle heuristic and the void depth test
  hash    a frame with the colour features from a multiresolution hash encoding
  batch   a planned batch of jobs of uneven size (one launch of the cicero_batch handle)

Scenes, MLPs, views and rays follow the distributions of the repository's synthetic workloads
(Gaussian blobs of density, smoothed noise as features, Xavier weights, orbiting cameras, rays from
a sphere aimed at the object), drawn on the GPU from the seed.
"""
import math
import random

import torch

from paper_2404_11852_gb300 import autograd as ag
from paper_2404_11852_gb300 import cicero as cc

DEV = "cuda"
PREC = {"bf16": cc.MLP_BF16, "f32": cc.MLP_FP32, "split": cc.MLP_FP32_SPLIT}


def listed():
    return [
        # the smallest call: an interactive preview of the small scene, bound by latency and launches
        dict(name="frame_bf16_64", kind="frame", prec="bf16", nx=64, ny=64, nz=64, C=12, f16=False, occ=0, blobs=8,
             w=64, h=64, S=64, march=False, brick=8),
        # an ordinary frame at an odd size, a grid that is no cube, 8 channels (no specialised path)
        dict(name="frame_bf16_odd", kind="frame", prec="bf16", nx=96, ny=113, nz=80, C=8, f16=False, occ=0, blobs=8,
             w=437, h=331, S=128, march=False, brick=8),
        # the benchmark's frame: 256^3 x 12 FP16 grid with a 32^3 occupancy mask, bricks as autotuned
        dict(name="frame_bf16_800", kind="frame", prec="bf16", nx=256, ny=256, nz=256, C=12, f16=True, occ=32,
             blobs=24, w=800, h=800, S=256, march=True, brick=4),
        # the same frame as the "plain FP32" render that the headline compares with (default options);
        # the largest case
        dict(name="frame_f32_800", kind="frame", prec="f32", nx=256, ny=256, nz=256, C=12, f16=True, occ=32,
             blobs=24, w=800, h=800, S=256, march=True, brick=8),
        # FP32-class quality on the tensor cores, an ordinary size
        dict(name="frame_split_320", kind="frame", prec="split", nx=160, ny=160, nz=160, C=12, f16=True, occ=32,
             blobs=24, w=320, h=320, S=192, march=True, brick=4),
        # one optimisation step of the training scene: 8192 rays x 256 samples, FP32 160^3 x 12 grid,
        # MSE loss, gradients of both grids and of the MLP
        dict(name="train_8192", kind="train", nx=160, ny=160, nz=160, C=12, f16=False, occ=0, blobs=8, R=8192, S=256),
        # fitting the grids only (pose refinement, frozen decoder), a ragged ray count, FP16 grid
        dict(name="grad_3001", kind="grad", nx=128, ny=128, nz=128, C=12, f16=True, occ=32, blobs=8, R=3001, S=192),
        # the headline: one SpaRW window of 16 targets at 800x800
        dict(name="window_800", kind="window", nx=256, ny=256, nz=256, C=12, f16=True, occ=32, blobs=24, w=800, h=800,
             S=256, march=True, views=16, brick=4, opaque=False),
        # a head-mounted trajectory on the small opaque scene: 15 frames in windows of 6 (the last ragged)
        dict(name="path_400", kind="path", nx=64, ny=64, nz=64, C=12, f16=False, occ=0, blobs=8, w=400, h=304, S=64,
             march=False, frames=15, window=6, brick=4, opaque=True),
        # one warped view at an odd size: phi heuristic, void test, depth output
        dict(name="warp_641", kind="warp", nx=128, ny=128, nz=128, C=12, f16=True, occ=32, blobs=8, w=641, h=479,
             S=192, march=True, phi=4.0),
        # hash-encoded colour features (8 levels x 2 FP16, 2^19 entries), 500x500
        dict(name="hash_500", kind="hash", nx=192, ny=192, nz=192, f16=True, occ=32, blobs=24, w=500, h=500, S=256,
             march=True, levels=8, log2=19, top=1024, brick=4),
        # a server's batch: nine views of three scenes, uneven sizes and sample counts
        dict(name="batch_9", kind="batch", C=12, f16=True, jobs=9, scenes=3, n_lo=96, n_hi=192, w_lo=128, w_hi=512,
             brick=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: sizes from the smallest listed to the largest, odd ones among them."""
    kind = rng.choice(["frame", "frame", "frame", "rays", "grad", "train", "window", "path", "warp", "hash", "batch"])
    f16 = rng.random() < 0.5
    # rows of the feature grid must be multiples of 16 bytes
    C = rng.choice([12, 12, 12, 12, 4, 8, 16])
    big = 256 if f16 else 176
    n = lambda: 2 * (_log(rng, 48, big) // 2)  # noqa: E731
    nx, ny, nz = (n(), n() + rng.randint(0, 1), n() + rng.randint(0, 1)) if rng.random() < 0.4 else (n(),) * 3
    g = dict(nx=nx, ny=ny, nz=nz, C=C, f16=f16, occ=rng.choice([0, 16, 32]), blobs=rng.randint(6, 24))
    S = rng.randint(33, 256)
    wh = lambda a, b: dict(w=_log(rng, a, b), h=_log(rng, a, b))  # noqa: E731
    march = rng.random() < 0.6
    if kind == "frame":
        prec = rng.choice(["bf16", "bf16", "f32", "split"])
        return dict(kind=kind, prec=prec, **g, **wh(40, 800 if prec == "bf16" else 400), S=S, march=march,
                    brick=rng.choice([4, 8]))
    if kind == "rays":
        return dict(kind=kind, prec=rng.choice(["bf16", "f32", "split"]), **g, R=_log(rng, 100, 20000), S=S,
                    brick=rng.choice([4, 8]))
    if kind in ("grad", "train"):
        if kind == "train":
            g["f16"] = False
            g.update({k: min(g[k], 176) for k in ("nx", "ny", "nz")})
        return dict(kind=kind, **g, R=_log(rng, 200, 8192), S=S)
    if kind == "window":
        return dict(kind=kind, **g, **wh(100, 500), S=S, march=march, views=rng.randint(1, 16), brick=4,
                    opaque=rng.random() < 0.5)
    if kind == "path":
        return dict(kind=kind, **g, **wh(100, 400), S=S, march=march, frames=rng.randint(5, 16),
                    window=rng.randint(2, 8), brick=4, opaque=rng.random() < 0.5)
    if kind == "warp":
        return dict(kind=kind, **g, **wh(64, 1000), S=S, march=march, phi=rng.choice([180.0, 4.0, 1.0]))
    if kind == "hash":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, f16=f16, occ=g["occ"], blobs=g["blobs"], **wh(64, 600), S=S,
                    march=march, levels=rng.choice([8, 8, rng.randint(4, 10)]), log2=rng.randint(14, 19),
                    top=rng.randint(256, 1024), brick=rng.choice([4, 8]))
    return dict(kind="batch", C=C, f16=f16, jobs=rng.randint(3, 12), scenes=rng.randint(1, 3), n_lo=64,
                n_hi=rng.randint(96, 176), w_lo=64, w_hi=rng.randint(160, 512), brick=rng.choice([4, 8]))


# ----------------------------------------------------------------------------------------------
# inputs


class _Draws:
    def __init__(self, seed):
        self.py = random.Random(int(seed))
        self.gen = torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFF)

    def uniform(self, shape, lo=-1.0, hi=1.0):
        return torch.rand(shape, generator=self.gen, device=DEV) * (hi - lo) + lo


def _smooth(a, axis):
    """One [1, 2, 1] / 4 pass, the edge vertex repeated."""
    n = a.shape[axis]
    lo = torch.cat([a.narrow(axis, 0, 1), a.narrow(axis, 0, n - 1)], axis)
    hi = torch.cat([a.narrow(axis, 1, n - 1), a.narrow(axis, n - 1, 1)], axis)
    return (lo + hi + 2.0 * a) * 0.25


def _cell_max(a, axis, R):
    N = a.shape[axis]
    parts = []
    for k in range(R):
        lo, hi = -(-k * (N - 1) // R), max((k + 1) * (N - 1) // R, -(-k * (N - 1) // R))
        parts.append(a.narrow(axis, lo, hi - lo + 1).amax(dim=axis, keepdim=True))
    return torch.cat(parts, axis)


def _grid(D, n, C, f16, occ, blobs, opaque=False):
    """cc.DeviceGrid of a blob scene on [-1, 1]^3; features None for C = 0."""
    ax = [torch.linspace(-1.0, 1.0, v, device=DEV, dtype=torch.float64) for v in n]
    raw = torch.zeros(n[2], n[1], n[0], device=DEV, dtype=torch.float64)
    for _ in range(blobs):
        mu = [D.py.uniform(-0.6, 0.6) for _ in range(3)]
        s, amp = D.py.uniform(0.06, 0.2), D.py.uniform(10.0, 40.0) * (25.0 if opaque else 1.0)
        gx, gy, gz = (torch.exp(-((a - m) ** 2) / (2 * s * s)) for a, m in zip(ax, mu))
        raw += (amp * gz)[:, None, None] * (gy[:, None] * gx[None, :])
    mask = None
    if occ:
        m = raw
        for a in range(3):
            m = _cell_max(m, a, occ)
        keep = math.ceil(0.15 * occ ** 3)
        mask = torch.zeros(occ ** 3, dtype=torch.uint8, device=DEV)
        mask[torch.topk(m.reshape(-1), keep).indices] = 1
        mask = mask.reshape(occ, occ, occ)
    t = torch.float16 if f16 else torch.float32
    feat = None
    if C:
        feat = D.uniform((n[2], n[1], n[0], C))
        for a in range(3):
            feat = _smooth(feat, a)
        feat = feat.to(t)
    return cc.DeviceGrid(raw.to(t), feat, occ=mask)


def _case_grid(D, c):
    return _grid(D, (c["nx"], c["ny"], c["nz"]), c.get("C", 0), c["f16"], c["occ"], c["blobs"], c.get("opaque", False))


def _mlp(D, C, grad=False):
    """Xavier weights and small biases, in_dim = C + 27 (4 frequencies of the direction)."""
    t = []
    for o, k in ((128, C + 27), (128, 128), (3, 128)):
        a = math.sqrt(6.0 / (o + k))
        t += [D.uniform((o, k), -a, a), D.uniform((o,), -0.1, 0.1)]
    if grad:
        t = [x.requires_grad_() for x in t]
    return cc.DeviceMlp(*t)


def _look_at(eye):
    """Camera-to-world rows (OpenCV axes) of a camera at eye that looks at the origin, z up."""
    unit = lambda v: [a / math.sqrt(sum(b * b for b in v)) for a in v]  # noqa: E731
    cross = lambda p, q: [p[1] * q[2] - p[2] * q[1], p[2] * q[0] - p[0] * q[2], p[0] * q[1] - p[1] * q[0]]  # noqa: E731
    z = unit([-a for a in eye])
    x = unit(cross(z, [0.0, 0.0, 1.0]))
    y = cross(z, x)
    return [[x[i], y[i], z[i], eye[i]] for i in range(3)]


def _orbit(w, h, az, el, radius=1.5, fov=40.0):
    a, e = math.radians(az), math.radians(el)
    c2w = _look_at([radius * math.cos(e) * math.cos(a), radius * math.cos(e) * math.sin(a), radius * math.sin(e)])
    f = (w / 2.0) / math.tan(math.radians(fov) / 2.0)
    return cc.camera(w, h, f, w / 2.0, h / 2.0, torch.tensor(c2w, dtype=torch.float32))


def _offset(cam, k, yaw=1.0, shift=0.005):
    """The pose k steps of a turning head from cam: yaw about its up axis, a step along its x axis."""
    m = torch.tensor(list(cam.c2w), dtype=torch.float64).reshape(3, 4)
    ang = math.radians(k * yaw)
    x, y, z, t = m.unbind(1)
    xr, zr = math.cos(ang) * x + math.sin(ang) * z, math.cos(ang) * z - math.sin(ang) * x
    out = torch.stack([xr, y, zr, t + k * shift * x], 1).float()
    return cc.camera(cam.width, cam.height, cam.f, cam.cx, cam.cy, out)


def _sampling(c):
    if not c.get("march", False):
        return cc.sampling(0.5, 2.5, c["S"], 0.0, 1e-3)
    return cc.sampling(0.0, 1e30, c["S"], 0.5 * 2.0 / (c["nx"] - 1), 1e-3)  # a slot every half voxel


def _rays(D, R):
    """Origins on the sphere of radius 1.5, aimed at points of [-0.5, 0.5]^3."""
    z, ph = D.uniform((R,)), D.uniform((R,), 0.0, 2.0 * math.pi)
    r = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    o = 1.5 * torch.stack([r * torch.cos(ph), r * torch.sin(ph), z], 1)
    d = D.uniform((R, 3), -0.5, 0.5) - o
    return o.contiguous(), (d / d.norm(dim=1, keepdim=True)).contiguous()


def _empty(*shape, dtype=torch.float32):
    return torch.empty(*shape, device=DEV, dtype=dtype)


def _options(c):
    """None (the default: FP32 MLP, bricks of 8) where that is what the case asks for."""
    prec = c.get("prec", "bf16")
    return None if prec == "f32" and c["brick"] == 8 else cc.options(PREC[prec], c["brick"])


def prepare(case, seed):
    c, D = case, _Draws(seed)
    kind = c["kind"]
    if kind == "batch":
        return _prepare_batch(c, D)
    grid = _case_grid(D, c)
    sd = _sampling(c)
    st = dict(case=c, grid=grid, sd=sd)
    if kind == "hash":
        levels = c["levels"]
        b = math.exp(math.log(c["top"] / 16) / (levels - 1))
        res = [int(16 * b ** i) for i in range(levels)]
        st["hash"] = cc.DeviceHashGrid(D.uniform((levels, 1 << c["log2"], 2)).half(), res, c["log2"])
        st["mlp"] = _mlp(D, 2 * levels)
    elif kind != "warp":
        st["mlp"] = _mlp(D, c["C"], grad=kind == "train")
    if kind in ("rays", "grad", "train"):
        R = c["R"]
        st["o"], st["d"] = _rays(D, R)
        if kind == "rays":
            st.update(opt=_options(c), rgb=_empty(R, 3), depth=_empty(R), acc=_empty(R))
            st["ws"] = cc.workspace(cc.cicero_render_workspace_size(grid.desc, R, sd, st["opt"]))
        elif kind == "grad":
            st["d_rgb"] = D.uniform((R, 3), -1e-3, 1e-3)
            st["ws"] = cc.workspace(cc.cicero_backward_workspace_size(grid.desc, R, sd))
        else:
            st["target"] = D.uniform((R, 3), 0.0, 1.0)
            st["density"] = grid.density.requires_grad_()
            st["features"] = grid.features.requires_grad_()
        return st
    w, h = c["w"], c["h"]
    R = w * h
    cam = st["cam"] = _orbit(w, h, D.py.uniform(0.0, 360.0), D.py.uniform(5.0, 40.0))
    opt = st["opt"] = _options(c) if kind != "warp" else None
    if kind == "frame":
        st.update(rgb=_empty(R, 3), depth=_empty(R), acc=_empty(R), n_steps=_empty(R, dtype=torch.int32))
        st["ws"] = cc.workspace(cc.cicero_render_workspace_size(grid.desc, R, sd, opt))
    elif kind == "hash":
        st.update(rgb=_empty(R, 3), depth=_empty(R))
        st["ws"] = cc.workspace(cc.cicero_render_hash_workspace_size(grid.desc, st["hash"].desc, R, sd, opt))
    elif kind == "warp":
        # a reference frame as a render leaves it: a smooth surface with steps, void around it
        ii, jj = (torch.arange(v, device=DEV, dtype=torch.float32) + 0.5 for v in (w, h))
        u, v = (ii / w - 0.5)[None, :], (jj / h - 0.5)[:, None]
        a, b = D.py.uniform(4.0, 9.0), D.py.uniform(4.0, 9.0)
        depth = 1.2 + 0.15 * torch.sin(a * u) * torch.cos(b * v) + 0.25 * (torch.sin(3 * a * u + b * v) > 0.6)
        depth = torch.where(u * u + v * v < 0.16, depth, torch.full_like(depth, math.inf)).reshape(-1).contiguous()
        st.update(ref_rgb=D.uniform((R, 3), 0.0, 1.0), ref_depth=depth, tgt=_offset(cam, 3), rgb=_empty(R, 3),
                  depth=_empty(R), mask=_empty(R, dtype=torch.uint8), idx=_empty(R, dtype=torch.int32),
                  n=_empty(1, dtype=torch.int32))
        st["ws"] = cc.workspace(cc.cicero_warp_workspace_size(st["tgt"]))
    elif kind == "window":
        V = c["views"]
        half = V // 2
        st["tgts"] = [_offset(cam, k - half if k < half else k - half + 1) for k in range(V)]
        st.update(ref_rgb=_empty(R, 3), ref_depth=_empty(R), rgb=[_empty(R, 3) for _ in range(V)],
                  depth=[_empty(R) for _ in range(V)], mask=[_empty(R, dtype=torch.uint8) for _ in range(V)],
                  idx=[_empty(R, dtype=torch.int32) for _ in range(V)], n=_empty(V, dtype=torch.int32))
        st["ws"] = cc.workspace(cc.cicero_render_workspace_size(grid.desc, R, sd, opt))
        st["ws_warp"] = cc.workspace(cc.cicero_warp_batch_workspace_size(st["tgts"]))
        # room for 64 samples of every target pixel (a quarter of the slots of a window)
        st["opt_h"] = cc.options(opt.precision, opt.brick, max_records=V * R * min(c["S"], 64))
        st["ws_h"] = cc.workspace(cc.cicero_render_workspace_size(grid.desc, V * R, sd, st["opt_h"]))
    else:  # path
        az, el = D.py.uniform(0.0, 360.0), D.py.uniform(5.0, 40.0)
        st["tgts"] = [_orbit(w, h, az + 0.5 * k, el) for k in range(c["frames"])]
        records = c["window"] * R * c["S"]
        ws = cc.workspace(cc.cicero_pipeline_workspace_size(grid.desc, cam, sd, opt, c["window"], records))
        st["pipe"] = cc.Pipeline(grid.desc, st["mlp"].desc, cam, sd, opt, c["window"], records, 180.0, ws)
        st["ref_stream"] = torch.cuda.Stream()
        st.update(rgb=[_empty(R, 3) for _ in st["tgts"]], depth=[_empty(R) for _ in st["tgts"]])
    return st


def _prepare_batch(c, D):
    scenes = []
    for _ in range(c["scenes"]):
        n = 2 * (D.py.randint(c["n_lo"], c["n_hi"]) // 2)
        scenes.append((n, _grid(D, (n, n, n), c["C"], c["f16"], 32, 24), _mlp(D, c["C"])))
    # the jobs' sizes are part of the case: the same for every seed
    size = random.Random(c["jobs"] * 1000003 + c["w_hi"])
    rows, specs = [], []
    for j in range(c["jobs"]):
        n, g, m = scenes[j % len(scenes)]
        w, h = (size.randint(c["w_lo"], c["w_hi"]) for _ in range(2))
        cam = _orbit(w, h, D.py.uniform(0.0, 360.0), D.py.uniform(5.0, 40.0))
        sd = _sampling(dict(march=True, S=size.choice([64, 128, 192, 256]), nx=n))
        rows.append((g.desc, m.desc, cam, sd, _empty(w * h, 3), _empty(w * h)))
        specs.append((g, m, cam, sd))
    jobs, opt = cc.jobs_array(rows), cc.options(cc.MLP_BF16, c["brick"])
    batch = cc.Batch(jobs, opt, cc.workspace(cc.cicero_batch_workspace_size(jobs, opt)))
    return dict(case=c, rows=rows, specs=specs, batch=batch)


# ----------------------------------------------------------------------------------------------
# one pass


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "batch":
        s["batch"].launch()
        return [[r[4], r[5]] for r in s["rows"]]
    g, sd = s["grid"].desc, s["sd"]
    if kind == "frame":
        cc.cicero_render(g, s["mlp"].desc, s["cam"], sd, s["opt"], s["rgb"], s["depth"], s["acc"], s["n_steps"], s["ws"])
        return dict(rgb=s["rgb"], depth=s["depth"], acc=s["acc"], n_steps=s["n_steps"])
    if kind == "rays":
        cc.cicero_render_rays(g, s["mlp"].desc, s["o"], s["d"], sd, s["opt"], s["rgb"], s["depth"], s["acc"], None,
                              s["ws"])
        return dict(rgb=s["rgb"], depth=s["depth"], acc=s["acc"])
    if kind == "grad":
        dd = torch.zeros(s["grid"].density.shape, device=DEV)
        df = torch.zeros(s["grid"].features.shape, device=DEV)
        cc.cicero_render_backward(g, s["mlp"].desc, s["o"], s["d"], sd, s["d_rgb"], dd, df, None, s["ws"])
        return dict(density=dd, features=df)
    if kind == "train":
        rgb = ag.render_rays(s["density"], s["features"], s["mlp"], s["o"], s["d"], _Spec(sd))
        loss = ((rgb - s["target"]) ** 2).mean()
        grads = torch.autograd.grad(loss, [s["density"], s["features"], *s["mlp"].t])
        return dict(rgb=rgb.detach(), loss=loss.detach(), grads=list(grads))
    if kind == "hash":
        cc.cicero_render_hash(g, s["hash"].desc, s["mlp"].desc, s["cam"], sd, s["opt"], s["rgb"], s["depth"], s["ws"])
        return dict(rgb=s["rgb"], depth=s["depth"])
    if kind == "warp":
        cc.cicero_warp(s["ref_rgb"], s["ref_depth"], s["cam"], s["tgt"], c["phi"], g, sd, s["rgb"], s["depth"],
                       s["mask"], s["idx"], s["n"], s["ws"])
        return dict(rgb=s["rgb"], depth=s["depth"], mask=s["mask"], n=s["n"])
    if kind == "window":
        cc.cicero_render(g, s["mlp"].desc, s["cam"], sd, s["opt"], s["ref_rgb"], s["ref_depth"], None, None, s["ws"])
        cc.cicero_warp_batch(s["ref_rgb"], s["ref_depth"], s["cam"], s["tgts"], 180.0, None, None, s["rgb"], s["depth"],
                             s["mask"], s["idx"], s["n"], s["ws_warp"])
        cc.cicero_render_holes_batch(g, s["mlp"].desc, s["tgts"], sd, s["opt_h"], s["idx"], s["n"],
                                     c["views"] * c["w"] * c["h"], s["rgb"], s["depth"], s["ws_h"])
        return dict(rgb=s["rgb"], depth=s["depth"], mask=s["mask"], n=s["n"])
    cur = torch.cuda.current_stream()
    s["ref_stream"].wait_stream(cur)
    s["pipe"].run(s["tgts"], s["rgb"], s["depth"], stream_tgt=cur, stream_ref=s["ref_stream"])
    return dict(rgb=s["rgb"], depth=s["depth"])


class _Spec:
    """Sampling as the autograd wrapper takes it."""

    def __init__(self, sd):
        self.near, self.far, self.n_samples, self.step = sd.near_t, sd.far_t, sd.n_samples, sd.step
        self.t_stop, self.bg, self.void_acc = sd.t_stop, tuple(sd.bg), sd.void_acc


# ----------------------------------------------------------------------------------------------
# what a pass cannot do without

# Share of a ray's slots that are composited, from the repository's scenes: about 0.39 for slots every
# half voxel inside the box (64.5 M of 163.8 M on the 800x800 frame), 0.45 for uniform slots in fog;
# two slots of a ray on opaque scenes.


def _samples(c, rays):
    if c.get("opaque"):
        return 2.0 * rays
    share = 0.39 if c.get("march") else 0.45
    return share * rays * min(c["S"], 256)


def work(case):
    c, kind = case, case["kind"]
    mlp = lambda C: 2 * ((C + 27) * 128 + 128 * 128 + 3 * 128)  # noqa: E731
    if kind == "batch":
        size = random.Random(c["jobs"] * 1000003 + c["w_hi"])
        rays = slots = 0
        for _ in range(c["jobs"]):
            w, h = (size.randint(c["w_lo"], c["w_hi"]) for _ in range(2))
            rays, slots = rays + w * h, slots + w * h * size.choice([64, 128, 192, 256])
        n = (c["n_lo"] + c["n_hi"]) / 2
        return dict(bytes=c["scenes"] * n ** 3 * (c["C"] + 1) * (2 if c["f16"] else 4) + 16 * rays,
                    flops=0.35 * slots * mlp(c["C"]))
    elem = 2 if c["f16"] else 4
    verts = c["nx"] * c["ny"] * c["nz"]
    grid = verts * elem * (1 + c.get("C", 0))
    if kind in ("rays", "grad", "train"):
        ns = _samples(c, c["R"])
        if kind == "rays":
            return dict(bytes=grid + 44 * c["R"], flops=ns * mlp(c["C"]))
        grads = 4 * verts * (1 + c["C"])  # written; the forward is computed again for them
        if kind == "grad":
            return dict(bytes=grid + grads + 36 * c["R"], flops=2 * ns * mlp(c["C"]))
        return dict(bytes=grid + grads + 60 * c["R"], flops=3 * ns * mlp(c["C"]))
    R = c["w"] * c["h"]
    if kind == "frame":
        return dict(bytes=grid + 24 * R, flops=_samples(c, R) * mlp(c["C"]))
    if kind == "hash":
        return dict(bytes=verts * elem + c["levels"] * 4 * (1 << c["log2"]) + 16 * R,
                    flops=_samples(c, R) * mlp(2 * c["levels"]))
    if kind == "warp":
        return dict(bytes=verts * 0 + 16 * R + 17 * R, flops=100 * R)
    V = c["views"] if kind == "window" else c["frames"]
    refs = 1 if kind == "window" else -(-V // c["window"])
    # a reference frame per window, and about an eighth of the target pixels as holes
    return dict(bytes=grid + 16 * R * refs + 16 * R * V, flops=_samples(c, R * (refs + V / 8)) * mlp(c["C"]))


# ----------------------------------------------------------------------------------------------
# the same values in 64 bits (plain torch)


def _trilinear(vol, i, f):
    """vol [Z][Y][X][K] at voxels i [n][3] and fractions f [n][3] (x, y, z)."""
    Z, Y, X, K = vol.shape
    flat = vol.reshape(-1, K)
    out = 0.0
    for q in range(8):
        x, y, z = i[:, 0] + (q & 1), i[:, 1] + ((q >> 1) & 1), i[:, 2] + (q >> 2)
        w = 1.0
        for a in range(3):
            w = w * (f[:, a] if (q >> a) & 1 else 1.0 - f[:, a])
        out = out + w[:, None] * flat[(z * Y + y) * X + x].double()
    return out


def _mlp64(t, x):
    h = torch.relu(x @ t[0].double().T + t[1].double())
    h = torch.relu(h @ t[2].double().T + t[3].double())
    return torch.sigmoid(h @ t[4].double().T + t[5].double())


def _encode64(d):
    parts = [d]
    for k in range(4):
        parts += [torch.sin(2.0 ** k * d), torch.cos(2.0 ** k * d)]
    return torch.cat(parts, 1)


def _hash64(hg, p):
    """Features of the multiresolution hash encoding at positions p of [-1, 1]^3."""
    u = ((p + 1.0) * 0.5).clamp(0.0, 1.0)
    T = hg.table.shape[1]
    out = []
    for lv in range(hg.table.shape[0]):
        N = hg.desc.res[lv]
        g = u * N
        i = g.floor().clamp(max=N - 1).long()
        f, acc = g - i, 0.0
        for q in range(8):
            x, y, z = (i[:, a] + ((q >> a) & 1) for a in range(3))
            if (N + 1) ** 3 <= T:
                at = x + (N + 1) * (y + (N + 1) * z)
            else:
                at = (x ^ (y * 2654435761) ^ (z * 805459861)) & (T - 1)
            w = 1.0
            for a in range(3):
                w = w * (f[:, a] if (q >> a) & 1 else 1.0 - f[:, a])
            acc = acc + w[:, None] * hg.table[lv][at].double()
        out.append(acc)
    return torch.cat(out, 1)


def _render64(grid, mlp_t, sd, o, d, hg=None):
    """(rgb, depth, acc) of rays o, d [R][3] in float64, as include/cicero.h defines them."""
    R, S = o.shape[0], sd.n_samples
    gd = grid.desc
    n = torch.tensor(list(gd.n), device=DEV, dtype=torch.float64)
    k = torch.arange(S, device=DEV, dtype=torch.float64) + 0.5
    if sd.step > 0:
        lo = torch.full((R,), float(sd.near_t), device=DEV, dtype=torch.float64)
        hi = torch.full((R,), float(sd.far_t), device=DEV, dtype=torch.float64)
        inv = 1.0 / d
        a, b = (-1.0 - o) * inv, (1.0 - o) * inv
        lo = torch.maximum(lo, torch.minimum(a, b).amax(1))
        hi = torch.minimum(hi, torch.maximum(a, b).amin(1))
        dt = float(sd.step)
        t = lo[:, None] + k * dt
        live = (t < hi[:, None]) & (lo < hi)[:, None]
    else:
        dt = (sd.far_t - sd.near_t) / S
        t = (sd.near_t + k * dt).expand(R, S)
        live = torch.ones(R, S, dtype=torch.bool, device=DEV)
    p = o[:, None, :] + t[..., None] * d[:, None, :]
    g = (p + 1.0) * 0.5 * (n - 1)
    live = live & ((g >= 0) & (g <= n - 1)).all(-1)
    r, s = live.nonzero(as_tuple=True)
    g = g[r, s]
    if gd.occ:
        Ro = gd.occ_res
        cell = (g * (Ro / (n - 1))).floor().clamp(max=Ro - 1).long()
        keep = grid.occ.reshape(-1)[(cell[:, 2] * Ro + cell[:, 1]) * Ro + cell[:, 0]] != 0
        r, s, g = r[keep], s[keep], g[keep]
    i = torch.minimum(g.floor(), n - 2).long()
    f = g - i
    raw = _trilinear(grid.density[..., None], i, f)[:, 0]
    sig = torch.nn.functional.softplus(raw + gd.act_shift)
    sdl = torch.zeros(R, S, device=DEV, dtype=torch.float64).index_put((r, s), sig * dt)
    cum = torch.cumsum(sdl, 1)
    T = torch.exp(-(cum - sdl))
    if sd.t_stop > 0:
        on = torch.cumsum((T < sd.t_stop).long(), 1) == 0
    else:
        on = torch.ones_like(T, dtype=torch.bool)
    w = T * -torch.expm1(-sdl) * on
    end = torch.exp(-(sdl * on).sum(1))
    use = on[r, s]
    r, s, i, f = r[use], s[use], i[use], f[use]
    ws, enc = w[r, s], _encode64(d)
    rgb = torch.zeros(R, 3, device=DEV, dtype=torch.float64)
    step = 1 << 20
    for at in range(0, r.numel(), step):
        q = slice(at, at + step)
        x = _hash64(hg, p[r[q], s[q]]) if hg is not None else _trilinear(grid.features, i[q], f[q])
        col = _mlp64(mlp_t, torch.cat([x, enc[r[q]]], 1))
        rgb = rgb.index_add(0, r[q], ws[q, None] * col)
    bg = torch.tensor(list(sd.bg), device=DEV, dtype=torch.float64)
    acc = w.sum(1)
    depth = torch.where(acc >= sd.void_acc, (w * t).sum(1) / acc, torch.full_like(acc, math.inf))
    return rgb + end[:, None] * bg, depth, acc


def _camera_rays64(cam):
    c2w = torch.tensor(list(cam.c2w), device=DEV, dtype=torch.float64).reshape(3, 4)
    i = torch.arange(cam.width, device=DEV, dtype=torch.float64) + 0.5
    j = torch.arange(cam.height, device=DEV, dtype=torch.float64) + 0.5
    dx = ((i - cam.cx) / cam.f).repeat(cam.height)
    dy = ((j - cam.cy) / cam.f).repeat_interleave(cam.width)
    v = torch.stack([dx, dy, torch.ones_like(dx)], 1) @ c2w[:, :3].T
    d = v / v.norm(dim=1, keepdim=True)
    return c2w[:, 3].expand_as(d).contiguous(), d


def _chunks64(grid, mlp_t, sd, o, d, hg=None):
    per = max(1, (1 << 22) // sd.n_samples)
    with torch.no_grad():
        got = [_render64(grid, mlp_t, sd, o[a:a + per], d[a:a + per], hg) for a in range(0, o.shape[0], per)]
    return [torch.cat(v) for v in zip(*got)]


class _As64:
    """A grid whose density and features are float64 leaves."""

    def __init__(self, grid):
        self.desc, self.occ = grid.desc, grid.occ
        self.density = grid.density.detach().double().requires_grad_()
        self.features = grid.features.detach().double().requires_grad_()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("window", "path", "warp"):
        return None  # which pixel a point lands on is decided in 32 bits: no 64-bit value
    s = prepare(case, seed)
    if kind == "batch":
        return [list(_chunks64(g, m.t, sd, *_camera_rays64(cam))[:2]) for g, m, cam, sd in s["specs"]]
    sd, m = s["sd"], s["mlp"].t
    if kind in ("frame", "hash"):
        rgb, depth, acc = _chunks64(s["grid"], m, sd, *_camera_rays64(s["cam"]), s["hash"] if kind == "hash" else None)
        return dict(rgb=rgb, depth=depth) if kind == "hash" else dict(rgb=rgb, depth=depth, acc=acc, n_steps=None)
    o, d = s["o"].double(), s["d"].double()
    if kind == "rays":
        rgb, depth, acc = _chunks64(s["grid"], m, sd, o, d)
        return dict(rgb=rgb, depth=depth, acc=acc)
    g64 = _As64(s["grid"])
    m64 = [t.detach().double().requires_grad_() for t in m]
    leaves = [g64.density, g64.features] + (m64 if kind == "train" else [])
    R, sums, rgbs = o.shape[0], None, []
    for a in range(0, R, 512):
        rgb = _render64(g64, m64, sd, o[a:a + 512], d[a:a + 512])[0]
        if kind == "grad":
            gr = s["d_rgb"][a:a + 512].double()
        else:
            gr = 2.0 * (rgb.detach() - s["target"][a:a + 512].double()) / (3 * R)
            rgbs.append(rgb.detach())
        got = torch.autograd.grad(rgb, leaves, gr)
        sums = list(got) if sums is None else [x + y for x, y in zip(sums, got)]
    if kind == "grad":
        return dict(density=sums[0], features=sums[1])
    rgb = torch.cat(rgbs)
    return dict(rgb=rgb, loss=((rgb - s["target"].double()) ** 2).mean(), grads=sums)
