"""The backward's FP32 fix-up (k_fwd_fix): samples whose ReLU decisions the tensor-core recompute lists as uncertain.
Features and direction are the same for every sample, and the biases put a third of the units of both layers
within the listing thresholds of zero, on a known side and ten times further from it than FP32 rounds: every
sample is listed, and its masks come from the fix-up."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -21  # the recompute's threshold, in units of ||W_n|| times the size of the inputs


@pytest.fixture(scope="module")
def cc():
    import torch
    assert torch.cuda.is_available()
    from paper_2404_11852_gb300 import cicero
    cicero.lib()
    return cicero


def scene(C, n_freq, side):
    """Grid, MLP; side: +1 or -1, the signs of the uncertain units' pre-activations as drawn or turned over.
    Half a threshold from zero: layer 1's FP32 chain errs by ~2^-24 of ||W_n|| ||x|| (its encoding of the
    direction z by ~3e-7 of its few inputs that are not exact), layer 2's by less than that of its inputs."""
    g = scenes.make_grid(24, C, 4, seed=30 + C)
    f = (0.1 * scenes.uniform(31 + C, C, -1.0, 1.0)).astype(np.float32)
    g.features[...] = f
    m = scenes.make_mlp(C, seed=32 + C, n_freq=n_freq, random_bias=True)
    d = np.array([0.0, 0.0, 1.0])
    x = np.concatenate([f.astype(np.float64), d] + [q for k in range(n_freq) for q in (np.sin(2.0 ** k * d), np.cos(2.0 ** k * d))])
    sgn = side * np.where(scenes.splitmix64(33 + C, 256) & np.uint64(1), 1.0, -1.0)
    w1, w2 = m.w1.astype(np.float64), m.w2.astype(np.float64)
    u = np.arange(128) % 3 == 1
    b = 0.5 * EPS * sgn[:128] * np.linalg.norm(w1, axis=1) * np.linalg.norm(x) - w1 @ x
    m.b1[u] = b[u]
    h = np.maximum(w1 @ x + m.b1, 0.0)
    scale = np.linalg.norm(h) + np.linalg.norm(x) * np.linalg.norm(w1)
    b = 0.5 * EPS * sgn[128:] * np.linalg.norm(w2, axis=1) * scale - w2 @ h
    m.b2[u] = b[u]
    return g, m


# rays x slots, all of them composited: one sample, part of a warp's four, and more than every warp of 200 SMs
# takes in its first turn, no multiple of four
@pytest.mark.parametrize("R,S", [(1, 1), (3, 2), (1301, 5)])
@pytest.mark.parametrize("C,n_freq,with_mlp", [(12, 4, False), (12, 4, True), (9, 0, True), (4, 1, False)])
def test_uncertain_decisions(cc, orc, R, S, C, n_freq, with_mlp):
    import torch
    o = (0.3 * scenes.uniform(40, 3 * R, -1.0, 1.0)).astype(np.float32).reshape(R, 3)
    d = np.tile(np.array([0.0, 0.0, 1.0], np.float32), (R, 1))
    sp = scenes.Sampling(near=0.0, far=0.5, n_samples=S, t_stop=0.0)
    grad = np.random.default_rng(R + C).standard_normal((R, 3)).astype(np.float32)
    g, m = scene(C, n_freq, 1)
    want = orc.backward(g, m, sp, grad, rays=(o, d), with_mlp=with_mlp)
    turned = orc.backward(g, scene(C, n_freq, -1)[1], sp, grad, rays=(o, d), with_mlp=with_mlp)
    assert np.abs(turned[1] - want[1]).max() > 1e-2 * np.abs(want[1]).max()  # wrong masks would show
    gd, md, sd = cc.DeviceGrid.from_host(g), cc.DeviceMlp.from_host(m), cc.sampling_from(sp)
    got = [torch.zeros(g.density.shape, device="cuda"), torch.zeros(g.features.shape, device="cuda"),
           torch.zeros(m.flat().size, device="cuda") if with_mlp else None]
    size = cc.cicero_backward_mlp_workspace_size if with_mlp else cc.cicero_backward_workspace_size
    ws = cc.workspace(size(gd.desc, R, sd))
    cc.cicero_profile_begin()
    cc.cicero_render_backward(gd.desc, md.desc, torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), sd,
                              torch.from_numpy(grad).cuda(), *got, ws)
    torch.cuda.synchronize()
    assert cc.cicero_profile_end()["gather_mlp"][1] == 2  # the recompute and the fix-up
    cc.cicero_workspace_status(ws)
    hdr = ws[:32].view(torch.int32).cpu().numpy()
    assert hdr[2] == R * S and hdr[4] == R * S  # composited, and all of them listed
    for a, b in zip(got, want):
        if a is not None:
            a = a.cpu().double().numpy().ravel()
            assert np.abs(a - np.ravel(b)).max() <= 1e-4 * np.abs(b).max()
