"""Packed voxels of an FP16 grid are made where they pay: by the rays that a call really has (holes are counted on
the device), their slots and their directions; the images have the same bits either way."""
import pytest

import scenes

pytestmark = pytest.mark.gpu

N, W, S = 64, 320, 128  # pack_min: 2.4 M + 0.92 x 64^3 = 2.64 M weighted slots without a mask, 2.53 M with one


@pytest.fixture(scope="module")
def cc():
    import torch
    assert torch.cuda.is_available()
    from paper_2404_11852_gb300 import cicero
    cicero.lib()
    return cicero


# azimuth, holes (None: the whole frame), occupancy mask, early stop, packed.  102,400 rays, nearly all of them
# through the box; 64 slots each with early stopping, ~100 without: 6.5 M and 10 M slots, times 1 - |dx| of ~0.94
# across x (azimuth 90) and ~0.08 along it (azimuth 0, elevation 20)
CASES = [(90.0, None, 0, 1e-3, True), (90.0, None, 16, 1e-3, True), (0.0, None, 0, 1e-3, False),
         (90.0, 1, 0, 1e-3, False), (90.0, 1024, 16, 0.0, False), (90.0, 0, 0, 1e-3, False),
         (90.0, 80000, 0, 0.0, True)]


@pytest.mark.parametrize("az,holes,occ,t_stop,packed", CASES)
def test_packing_follows_the_rays(cc, az, holes, occ, t_stop, packed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(5)
    dens = (torch.rand((N, N, N), generator=gen, device="cuda") * 4 - 6).half()
    feat = (torch.rand((N, N, N, 4), generator=gen, device="cuda") * 2 - 1).half()
    mask = torch.ones((occ,) * 3, dtype=torch.uint8, device="cuda") if occ else None
    g, m = cc.DeviceGrid(dens, feat, occ=mask), cc.DeviceMlp.from_host(scenes.make_mlp(4, seed=3))
    cd = cc.camera_from(scenes.orbit_camera(W, W, az_deg=az, el_deg=20.0))
    sd, opt, R = cc.sampling(0.5, 2.5, S, 0.0, t_stop), cc.options(cc.MLP_BF16, 4), W * W
    need = cc.cicero_render_workspace_size(g.desc, R, sd, opt)
    voxels = 16 * N ** 3
    got = []
    for bytes_ in (need, need - voxels):
        ws = cc.workspace(bytes_)
        tail = ws[need - voxels:need]
        tail.fill_(0xA5)
        rgb, depth = torch.zeros(R, 3, device="cuda"), torch.zeros(R, device="cuda")
        if holes is None:
            cc.cicero_render(g.desc, m.desc, cd, sd, opt, rgb, depth, None, None, ws)
        else:
            idx = torch.arange(R, device="cuda", dtype=torch.int32)
            n = torch.tensor([holes], device="cuda", dtype=torch.int32)
            cc.cicero_render_holes(g.desc, m.desc, cd, sd, opt, idx, n, R, rgb, depth, ws)
        cc.cicero_workspace_status(ws)
        if bytes_ == need:
            assert bool((tail != 0xA5).any()) == packed
        got.append((rgb, depth))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


def test_workspaces_without_the_voxels(cc):
    """The autotuner and the pipeline take a workspace without room for the packed voxels, as a render does, and
    give the same images; one smaller still is refused."""
    import torch
    n, w, S, window = 48, 160, 64, 3
    g = cc.DeviceGrid.from_host(scenes.make_grid(n, 4, 6, seed=7, dtype="float16"))
    m = cc.DeviceMlp.from_host(scenes.make_mlp(4, seed=8))
    cams = [scenes.orbit_camera(w, w, az_deg=60.0 + k) for k in range(5)]
    cds = [cc.camera_from(c) for c in cams]
    sd, R, voxels = cc.sampling(0.5, 2.5, S, 0.0, 1e-3), w * w, (16 * n ** 3 + 255) // 256 * 256
    need = max(cc.cicero_render_workspace_size(g.desc, R, sd, cc.options(cc.MLP_BF16, b)) for b in (4, 8, 16))
    rgb, depth = torch.empty(R, 3, device="cuda"), torch.empty(R, device="cuda")
    best, ms = cc.cicero_autotune_brick(g.desc, m.desc, cds[0], sd, cc.MLP_BF16, rgb, depth, cc.workspace(need - voxels))
    assert best in (4, 8, 16) and all(t > 0 for t in ms.values())
    opt, records = cc.options(cc.MLP_BF16, 4), window * R * S
    need = cc.cicero_pipeline_workspace_size(g.desc, cds[0], sd, opt, window, records)
    out = []
    for bytes_ in (need, need - 3 * voxels):
        frames = [torch.empty(R, 3, device="cuda") for _ in cds], [torch.empty(R, device="cuda") for _ in cds]
        ws = cc.workspace(bytes_)
        pipe = cc.Pipeline(g.desc, m.desc, cds[0], sd, opt, window, records, 180.0, ws)
        pipe.run(cds, *frames)
        torch.cuda.synchronize()
        out.append(frames)
    for a, b in zip(out[0][0] + out[0][1], out[1][0] + out[1][1]):
        assert torch.equal(a, b)
    with pytest.raises(cc.CiceroError):
        cc.Pipeline(g.desc, m.desc, cds[0], sd, opt, window, records, 180.0, cc.workspace(need - 3 * voxels - 256))
