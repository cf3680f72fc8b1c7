"""Calls queued right behind the kernels that write their inputs, and before the ones that overwrite them: every
call sees the parameters and inputs as they were at its place on the stream."""
import pytest

import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cc():
    import torch
    assert torch.cuda.is_available()
    from paper_2404_11852_gb300 import cicero
    cicero.lib()
    return cicero


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_updates_between_calls(cc, precision):
    import torch
    C, w, M = 12, 48, 300
    g = cc.DeviceGrid.from_host(scenes.make_grid(32, C, 4, seed=1))
    live, steps = cc.DeviceMlp.from_host(scenes.make_mlp(C, seed=2)), 6
    sets = [cc.DeviceMlp.from_host(scenes.make_mlp(C, seed=3 + k, random_bias=True)).t for k in range(steps)]
    xs = [torch.rand(M, C + 27, device="cuda") * 2 - 1 for _ in sets]
    x = torch.empty_like(xs[0])
    cam = scenes.orbit_camera(w, w, sampling=scenes.sampling_uniform(32))
    cd, sd, opt = cc.camera_from(cam), cc.sampling_from(cam.sampling), cc.options(precision, 4)
    ws = cc.workspace(cc.cicero_render_workspace_size(g.desc, w * w, sd, opt))
    ws_e = cc.workspace(cc.cicero_mlp_eval_workspace_size(M))

    def go(wait):
        out = []
        for new, xi in zip(sets, xs):
            c, rgb, depth = torch.empty(M, 3, device="cuda"), torch.empty(w * w, 3, device="cuda"), torch.empty(w * w, device="cuda")
            x.copy_(xi)
            torch._foreach_copy_(live.t, new)
            if wait:
                torch.cuda.synchronize()
            if precision < 2:
                cc.cicero_mlp_eval(live.desc, x, precision, c, ws_e)
                out.append(c)
            cc.cicero_render(g.desc, live.desc, cd, sd, opt, rgb, depth, None, None, ws)
            out += [rgb, depth]
            if wait:
                torch.cuda.synchronize()
            for t in live.t:
                t.fill_(1e3)
        torch.cuda.synchronize()
        return out

    for a, b in zip(go(True), go(False)):
        assert torch.equal(a, b)
