"""Feature-channel layouts of the gather + MLP kernels against the FP64 oracle.  BF16 (2e-2, the path's
tolerance): every specialised channel count and the general kernel, with the features from staged bricks
and, where those leave room for fewer tiles in flight, from global memory.  FP32 and split BF16: the
pipelined tensor-core kernel, from a single tile to several per SM."""
import numpy as np
import pytest

import scenes
from helpers import check_render, gpu_render

pytestmark = pytest.mark.gpu

TOL16, PSNR16 = 2e-2, 45.0


@pytest.fixture(scope="module")
def cc():
    import torch
    assert torch.cuda.is_available()
    from paper_2404_11852_gb300 import cicero
    cicero.lib()
    return cicero


# (channels, frequencies, grid type, brick): bricks of 4 are staged; bricks of 8 of an FP32 grid with 8
# or more channels are gathered from global memory (two staged bricks at most would fit).  C + 3 + 6
# n_freq = 48 leaves no column for the folded bias.
LAYOUTS = [(4, 4, np.float16, 4), (4, 4, np.float32, 8), (8, 4, np.float32, 8), (8, 4, np.float16, 4),
           (12, 4, np.float32, 8), (16, 4, np.float32, 8), (16, 4, np.float16, 8), (21, 4, np.float32, 8),
           (6, 4, np.float16, 4), (1, 7, np.float32, 4), (3, 7, np.float32, 8), (5, 0, np.float32, 4),
           (13, 2, np.float32, 8)]


@pytest.mark.parametrize("C,n_freq,dtype,brick", LAYOUTS)
def test_bf16_channel_layouts(cc, orc, C, n_freq, dtype, brick):
    g = scenes.make_grid(32, C, 4, seed=300 + C, dtype=dtype)
    m = scenes.make_mlp(C, seed=400 + C, n_freq=n_freq, random_bias=True)
    cam = scenes.orbit_camera(31, 27, az_deg=50.0, sampling=scenes.sampling_uniform(48))
    ref = orc.render(g, m, cam.sampling, cam=cam)
    check_render(gpu_render(cc, g, m, cam, cam.sampling, cc.MLP_BF16, brick), ref, TOL16, psnr_min=PSNR16)


@pytest.mark.parametrize("C,brick", [(8, 8), (5, 4)])
def test_batch_channel_layouts(cc, C, brick):
    """A batch of another channel count renders its jobs bit for bit as single calls do."""
    import torch
    g = cc.DeviceGrid.from_host(scenes.make_grid(32, C, 4, seed=500 + C))
    m = cc.DeviceMlp.from_host(scenes.make_mlp(C, seed=501, random_bias=True))
    cams = [scenes.orbit_camera(33, 21, az_deg=a, sampling=scenes.sampling_uniform(40)) for a in (0.0, 90.0)]
    sd, opt = cc.sampling_from(cams[0].sampling), cc.options(cc.MLP_BF16, brick)
    cds = [cc.camera_from(c) for c in cams]
    out = [(torch.empty(33 * 21, 3, device="cuda"), torch.empty(33 * 21, device="cuda")) for _ in cams]
    jobs = cc.jobs_array([(g.desc, m.desc, cd, sd, *o) for cd, o in zip(cds, out)])
    b = cc.Batch(jobs, opt, cc.workspace(cc.cicero_batch_workspace_size(jobs, opt)))
    b.launch()
    b.status()
    for cam, (rgb, depth) in zip(cams, out):
        one = gpu_render(cc, None, None, cam, cam.sampling, cc.MLP_BF16, brick, dev_grid=g, dev_mlp=m)
        assert (rgb.cpu().numpy().astype(np.float64) == one["rgb"]).all()
        assert (depth.cpu().numpy().astype(np.float64) == one["depth"]).all()


# |d rgb| <= sum of weights (<= 1) x sigmoid' (1/4) x |d z3|.  FP32: six products of three BF16 parts leave
# ~2^-24 of each term, and the accumulations ~11 x 2^-24 of a sum of a few units: ~1e-6, beside the march's
# ~3e-7; split BF16 leaves ~2^-17 of each term: ~1.5e-5.
TOL_SPLIT = {0: 5e-6, 2: 2e-5}


@pytest.mark.parametrize("precision,C,n_freq,dtype", [
    (0, 12, 4, np.float16), (0, 12, 4, np.float32), (0, 8, 4, np.float16), (0, 21, 4, np.float32), (0, 1, 7, np.float32),
    (0, 5, 0, np.float32), (0, 13, 2, np.float32), (2, 12, 4, np.float16), (2, 16, 4, np.float32), (2, 3, 7, np.float32),
    (2, 6, 4, np.float16)])
def test_split_channel_layouts(cc, orc, precision, C, n_freq, dtype):
    g = scenes.make_grid(32, C, 4, seed=600 + C, dtype=dtype)
    m = scenes.make_mlp(C, seed=700 + C, n_freq=n_freq, random_bias=True)
    cam = scenes.orbit_camera(29, 33, az_deg=70.0, sampling=scenes.sampling_uniform(48))
    ref = orc.render(g, m, cam.sampling, cam=cam)
    check_render(gpu_render(cc, g, m, cam, cam.sampling, precision, 4), ref, TOL_SPLIT[precision])


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("side,n_samples", [(1, 1), (2, 40), (12, 16), (40, 40), (120, 64)])
def test_split_tile_counts(cc, orc, precision, side, n_samples):
    """Tiles per SM from none or one to several, bricks of 16 (full tiles) and 4 (ragged ones)."""
    g, m = scenes.make_grid(48, 12, 6, seed=81), scenes.make_mlp(12, seed=82, random_bias=True)
    cam = scenes.orbit_camera(side, side, az_deg=20.0, sampling=scenes.sampling_uniform(n_samples))
    pix = (scenes.splitmix64(83, 200) % np.uint64(side * side)).astype(np.int32) if side > 40 else None
    ref = orc.render(g, m, cam.sampling, cam=cam, pix=pix)
    for brick in (4, 8):
        out = gpu_render(cc, g, m, cam, cam.sampling, precision, brick)
        if pix is not None:
            out = {k: v[pix] for k, v in out.items()}
        check_render(out, ref, TOL_SPLIT[precision])


@pytest.mark.parametrize("C,dtype,with_mlp", [(4, np.float32, False), (8, np.float16, True), (16, np.float32, True),
                                              (3, np.float32, True)])
def test_backward_masks_and_fixup(cc, orc, C, dtype, with_mlp):
    """The recompute's ReLU masks, its FP32 fix-up and the staged operands at other channel counts: every
    gradient within 1e-4 relative of the oracle's (a single flipped mask moves d_features by ~1e-3)."""
    import torch
    g = scenes.make_grid(32, C, 4, seed=800 + C, dtype=dtype)
    m = scenes.make_mlp(C, seed=810 + C, random_bias=True)
    o, d = scenes.random_rays(300, seed=820 + C)
    sp = scenes.Sampling(near=0.5, far=2.5, n_samples=40, t_stop=0.0)
    out = orc.render(g, m, sp, rays=(o, d))
    grad = np.random.default_rng(C).standard_normal((300, 3))
    grad[out["amb"]] = 0.0
    want = orc.backward(g, m, sp, grad, rays=(o, d), with_mlp=with_mlp)
    gd, md, sd = cc.DeviceGrid.from_host(g), cc.DeviceMlp.from_host(m), cc.sampling_from(sp)
    got = [torch.zeros(g.density.shape, device="cuda"), torch.zeros(g.features.shape, device="cuda"),
           torch.zeros(m.flat().size, device="cuda") if with_mlp else None]
    size = cc.cicero_backward_mlp_workspace_size if with_mlp else cc.cicero_backward_workspace_size
    ws = cc.workspace(size(gd.desc, 300, sd))
    cc.cicero_render_backward(gd.desc, md.desc, torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), sd,
                              torch.from_numpy(grad.astype(np.float32)).cuda(), *got, ws)
    cc.cicero_workspace_status(ws)
    for a, b in zip(got, want):
        if a is not None:
            a = a.cpu().double().numpy().ravel()
            assert np.abs(a - np.ravel(b)).max() <= 1e-4 * np.abs(b).max()


@pytest.mark.parametrize("N,brick,side", [(9, 4, 7), (33, 4, 40), (66, 4, 33), (130, 4, 24)])
def test_ray_index_table_scan(cc, N, brick, side):
    """The table from one scan block (1024 bricks) to several dozen, and tiles that end inside a brick:
    offsets and samples are consistent, and every sample of a brick appears once."""
    import torch
    g = scenes.make_grid(N, 4, 3, seed=900 + N)
    cam = scenes.orbit_camera(side, side, az_deg=35.0, sampling=scenes.sampling_uniform(64, t_stop=0.0))
    gd, cd, sd = cc.DeviceGrid.from_host(g), cc.camera_from(cam), cc.sampling_from(cam.sampling)
    opt = cc.options(cc.MLP_FP32, brick)
    nb = (-(-(N - 1) // brick)) ** 3
    offs = torch.full((nb + 1,), -1, dtype=torch.int32, device="cuda")
    smp = torch.full((side * side * 64,), -1, dtype=torch.int32, device="cuda")
    ws = cc.workspace(cc.cicero_build_rit_workspace_size(gd.desc, cd, sd, opt))
    assert cc.cicero_build_rit(gd.desc, cd, sd, opt, offs, smp, ws) == nb
    cc.cicero_workspace_status(ws)
    o, n = offs.cpu().numpy(), None
    hdr = ws[:16].view(torch.int32).cpu().numpy()
    n = int(hdr[2])
    assert o[0] == 0 and o[-1] == n and (np.diff(o) >= 0).all()
    assert int(hdr[1]) == int((-(-np.diff(o) // 128)).sum())  # tiles
    got = smp.cpu().numpy()[:n]
    assert len(np.unique(got)) == n and got.min() >= 0
    # the brick of each sample, from its position in FP64; samples within rounding of a face may differ
    ray, slot = got // 64, got % 64
    c2w = cam.c2w.astype(np.float64)
    u = np.stack([(ray % side + 0.5 - cam.cx) / cam.f, (ray // side + 0.5 - cam.cy) / cam.f, np.ones(n)], 1)
    d = u @ c2w[:, :3].T
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    p = c2w[:, 3] + (0.5 + (slot + 0.5) * (2.0 / 64))[:, None] * d
    v = np.minimum(np.floor((p + 1.0) * 0.5 * (N - 1)), N - 2).astype(int) // brick
    k = -(-(N - 1) // brick)
    want = (v[:, 2] * k + v[:, 1]) * k + v[:, 0]
    assert (want == np.repeat(np.arange(nb), np.diff(o))).mean() > 0.999


@pytest.mark.parametrize("w,h,void", [(1, 1, True), (37, 29, False), (64, 64, True), (129, 130, True), (4096, 3, False)])
def test_warp_hole_list(cc, orc, w, h, void):
    """Hole counting and listing from a single chunk of 4096 pixels to several, ragged ones among them."""
    import torch
    cam = scenes.orbit_camera(w, h, az_deg=10.0, sampling=scenes.sampling_uniform(32))
    tgt = scenes.offset_camera(cam, 3)
    g = scenes.make_grid(24, 4, 3, seed=950)
    rng = np.random.default_rng(w * h)
    rgb = rng.random((w * h, 3), dtype=np.float32)
    depth = np.where(rng.random(w * h) < 0.3, np.inf, 1.0 + 0.3 * rng.random(w * h)).astype(np.float32)
    want = orc.warp(rgb, depth, cam, tgt, void_grid=g if void else None, void_sampling=cam.sampling if void else None)
    gd, sd = cc.DeviceGrid.from_host(g), cc.sampling_from(cam.sampling)
    out = [torch.empty(w * h, 3, device="cuda"), torch.empty(w * h, device="cuda"),
           torch.empty(w * h, dtype=torch.uint8, device="cuda"), torch.empty(w * h, dtype=torch.int32, device="cuda"),
           torch.empty(1, dtype=torch.int32, device="cuda")]
    tc = cc.camera_from(tgt)
    cc.cicero_warp(torch.from_numpy(rgb).cuda(), torch.from_numpy(depth).cuda(), cc.camera_from(cam), tc, 180.0,
                   gd.desc if void else None, sd if void else None, *out, cc.workspace(cc.cicero_warp_workspace_size(tc)))
    assert (out[2].cpu().numpy() == want["mask"]).all()
    n = int(out[4].item())
    assert n == want["n_holes"]
    assert (out[3].cpu().numpy()[:n] == np.flatnonzero(want["mask"] == 1)).all()
    assert (out[0].cpu().numpy() == want["rgb"].astype(np.float32)).all()


@pytest.mark.parametrize("n,occ,precision", [((2, 2, 2), 0, 1), ((6, 3, 35), 0, 0), ((34, 17, 9), 5, 1),
                                             ((18, 40, 33), 64, 1), ((66, 33, 20), 16, 2), ((50, 51, 52), 1, 0)])
def test_packed_density_is_the_same(cc, n, occ, precision):
    """The march over packed voxels (k_pack) gives the bits of the march over the density array, which a
    workspace without room for the voxels takes: odd sizes, cells larger and smaller than voxels."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(sum(n) + occ)
    dens = (torch.rand((n[2], n[1], n[0]), generator=gen, device="cuda") * 12 - 4).half()
    feat = (torch.rand((n[2], n[1], n[0], 4), generator=gen, device="cuda") * 2 - 1).half()
    mask = (torch.rand((occ,) * 3, generator=gen, device="cuda") < 0.4).to(torch.uint8) if occ else None
    g, m = cc.DeviceGrid(dens, feat, occ=mask), cc.DeviceMlp.from_host(scenes.make_mlp(4, seed=3))
    cam = scenes.orbit_camera(90, 61, az_deg=33.0)
    cd, opt = cc.camera_from(cam), cc.options(precision, 4)
    R = 90 * 61
    for sd in (cc.sampling(0.5, 2.5, 300, 0.0, 1e-3), cc.sampling(0.0, 1e30, 120, 0.03, 0.0)):
        need = cc.cicero_render_workspace_size(g.desc, R, sd, opt)
        out = []
        for bytes_ in (need, need - 256):
            ws = cc.workspace(bytes_)
            o = [torch.empty(R, 3, device="cuda"), torch.empty(R, device="cuda"), torch.empty(R, device="cuda"),
                 torch.empty(R, dtype=torch.int32, device="cuda")]
            cc.cicero_profile_begin()
            n0 = cc.cicero_launch_count()
            cc.cicero_render(g.desc, m.desc, cd, sd, opt, *o, ws)
            launches = cc.cicero_launch_count() - n0
            cc.cicero_profile_end()
            cc.cicero_workspace_status(ws)
            out.append((launches, o))
        assert out[0][0] == out[1][0] + 1  # one kernel more: the packing
        for a, b in zip(out[0][1], out[1][1]):
            assert torch.equal(a, b)
        with pytest.raises(cc.CiceroError):  # without the voxels the workspace may not shrink any further
            cc.cicero_render(g.desc, m.desc, cd, sd, opt, *out[0][1], cc.workspace(need - 512 - 16 * n[0] * n[1] * n[2]))
