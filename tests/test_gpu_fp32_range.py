"""FP32 renders where an operand of the MLP has no BF16 parts: infinities, and finite values above BF16's
largest (3.396e38 and up round to infinity).  The colours are those of the FP32 chain (the oracle's in 64
bits), for the samples that reach such operands and for the others of the same call."""
import numpy as np
import pytest

import scenes
from helpers import check_render, gpu_render

pytestmark = pytest.mark.gpu

BIG, SMALL = np.float32(3.398e38), np.float32(2e-38)  # between BF16's and FP32's largest; their product is ~7
# Pre-activations up to ~12, ~50 roundings of 2^-24 of one, walking: 5e-6.  In the cells where a feature steps
# by 6.8 / weight, a voxel fraction's error of 4e-6 (FP32 positions over 15.5 cells a unit) moves every unit
# of layer 1 by 2.5e-5.  Through two layers of norm ~1.4 each 5e-5 and the sigmoid (1/4) 1.3e-5, three of which:
TOL = 4e-5


@pytest.fixture(scope="module")
def cc():
    import torch
    assert torch.cuda.is_available()
    from paper_2404_11852_gb300 import cicero
    cicero.lib()
    return cicero


def signs(seed, n):
    return np.where(scenes.splitmix64(seed, n) & np.uint64(1), 1, -1).astype(np.float32)


def scene(kind, C):
    g = scenes.make_grid(32, C, 4, seed=900 + C, dtype=np.float16 if kind == "inf_feature" and C == 12 else np.float32)
    m = scenes.make_mlp(C, seed=910 + C, random_bias=True)
    half = np.arange(32) >= 16  # the upper half along x, so that a tile's samples differ
    if kind == "big_feature":
        g.features[:, :, half, 0] = BIG
        g.features[:, :, ~half, 0] = 0.0
        m.w1[:, 0] = SMALL * signs(1, 128)
    elif kind == "big_w1":
        g.features[..., 0] = SMALL
        m.w1[:, 0] = BIG * signs(2, 128)
    elif kind in ("big_h1", "big_w2"):
        m.w1[5, :] = 0.0
        m.b1[5] = BIG if kind == "big_h1" else SMALL
        m.w2[:, 5] = (SMALL if kind == "big_h1" else BIG) * signs(3, 128)
    elif kind == "inf_feature":  # one unit of layer 1 is infinite, the others 0; then all of layer 2
        g.features[:, :, half, 0] = np.inf
        m.w1[:, 0] = -np.abs(m.w1[:, 0]) - 0.01
        m.w1[0, 0] = 0.5
        m.w2[:, 0] = 0.25
        m.w3[:] = np.abs(m.w3) + 0.01
        m.w3[1] *= -1.0
    elif kind == "nan_feature":
        g.features[:, :, half, 0] = np.nan
    elif kind == "nan_weight":  # a unit of NaNs is 0 behind the ReLU
        m.w1[0, 2] = m.w1[9, 1] = m.w2[0, 7] = m.w2[33, 3] = np.nan
    return g, m


def on_a_face(cam):
    """Rays with a sample in the upper half of the 32^3 grid along x, or on its edge, whose voxel coordinates
    come within 1e-5 of a whole number (FP32 positions err by ~4e-6 of a cell): whether its fraction is 0, which
    makes a NaN of an infinity, and which cell it falls into is decided by rounding."""
    i, j = np.meshgrid(np.arange(cam.width) + 0.5, np.arange(cam.height) + 0.5)
    d = np.stack([(i - cam.cx) / cam.f, (j - cam.cy) / cam.f, np.ones_like(i)], -1).reshape(-1, 3) @ cam.c2w[:, :3].T
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    sp = cam.sampling
    t = sp.near + (np.arange(sp.n_samples) + 0.5) * (sp.far - sp.near) / sp.n_samples
    g = (cam.c2w[None, None, :, 3] + t[None, :, None] * d[:, None, :] + 1.0) * 15.5
    near = (np.abs(g - np.round(g)) < 1e-5).any(-1) & ((g > -1e-5) & (g < 31 + 1e-5)).all(-1) & (g[..., 0] > 15 - 1e-5)
    return near.any(1)


@pytest.mark.parametrize("C", [12, 5])
@pytest.mark.parametrize("kind", ["big_feature", "big_w1", "big_h1", "big_w2", "inf_feature", "nan_feature",
                                  "nan_weight"])
def test_fp32_operands_without_bf16_parts(cc, orc, kind, C):
    g, m = scene(kind, C)
    cam = scenes.orbit_camera(31, 23, az_deg=40.0, sampling=scenes.sampling_uniform(40))
    ref = orc.render(g, m, cam.sampling, cam=cam)
    assert np.isfinite(ref["rgb"]).all()
    out = gpu_render(cc, g, m, cam, cam.sampling, cc.MLP_FP32, 4)
    if kind in ("inf_feature", "nan_feature"):
        keep = ~on_a_face(cam)
        assert (~keep).sum() <= 3
        out, ref = ({k: v[keep] for k, v in o.items()} for o in (out, ref))
    check_render(out, ref, TOL)


@pytest.mark.parametrize("kind", ["big_feature", "inf_feature"])
def test_wide_backward_recompute(cc, orc, kind):
    """The backward of more than 16 channels takes its colours from the same kernel: the density's gradient."""
    import torch
    C, R = 20, 200
    g, m = scene(kind, C)
    o, d = scenes.random_rays(R, seed=77)
    sp = scenes.Sampling(near=0.5, far=2.5, n_samples=24, t_stop=0.0)
    grad = np.random.default_rng(5).standard_normal((R, 3)).astype(np.float32)
    want = orc.backward(g, m, sp, grad, rays=(o, d))[0].ravel()
    assert np.isfinite(want).all()
    gd, md, sd = cc.DeviceGrid.from_host(g), cc.DeviceMlp.from_host(m), cc.sampling_from(sp)
    dd, df = torch.zeros(g.density.shape, device="cuda"), torch.zeros(g.features.shape, device="cuda")
    ws = cc.workspace(cc.cicero_backward_workspace_size(gd.desc, R, sd))
    cc.cicero_render_backward(gd.desc, md.desc, torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), sd,
                              torch.from_numpy(grad).cuda(), dd, df, None, ws)
    cc.cicero_workspace_status(ws)
    assert np.abs(dd.cpu().double().numpy().ravel() - want).max() <= 1e-3 * np.abs(want).max()  # the path's tolerance
