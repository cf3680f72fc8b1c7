"""Feature-channel layouts of the BF16 gather + MLP kernels against the FP64 oracle (2e-2, the path's
tolerance): every specialised channel count and the general kernel, with the features from staged bricks
and, where those leave room for fewer tiles in flight, from global memory."""
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
