"""Forwards and renders whose instance count outgrows, fits or undercuts the buffers an earlier one left:
the same bits as from a rasterizer or session of its own."""
import numpy as np
import pytest

import gsinputs as gi

pytestmark = pytest.mark.gpu

CASES = [(300, 64, 48), (6000, 256, 256), (200, 64, 48), (30000, 320, 200), (6000, 256, 256), (1, 33, 40)]


def test_raster_forwards():
    import torch
    import paper_2503_13086_gb300 as gs
    shared = gs.Raster()
    for n, w, h in CASES:
        p = torch.tensor(gi.cube_scene(n, seed=n), device="cuda")
        cam = gi.identity_camera(w, h, 1.0 * w)
        tgt = torch.tensor(gi.uniform_target(w, h, 1).reshape(-1), device="cuda")
        res = []
        for ras in (gs.Raster(), shared):
            o = ras.forward(p, n, [cam])
            loss, d = ras.loss(o["image"], tgt)
            g, _ = ras.backward(p, o["image"], o["last"], d)
            res.append([o[k].cpu().numpy() for k in ("image", "T", "last", "gp")] + [o["pairs"], loss, g.cpu().numpy()])
        for a, b in zip(*res):
            assert np.array_equal(a, b), (n, w, h)
    shared.close()


def test_renders_between_steps():
    import paper_2503_13086_gb300 as gs
    n = 6000
    p = gi.cube_scene(n, seed=3)
    big, small = gi.identity_camera(320, 256, 300.0), gi.identity_camera(48, 33, 40.0)

    def field():
        f = gs.Field(scene_extent=1.0, tiling=(16, 16, 256))
        f.set_gaussians(p[:, :n])
        return f, f.add_image(small, gi.uniform_target(48, 33, 2))

    a, img = field()
    b, _ = field()
    got = []
    for cam in (small, big, small):  # the second outgrows what the small view's steps left
        a.optimize_step([img])
        got.append(a.render(cam).cpu().numpy())
    for k, cam in enumerate((small, big, small)):
        b.optimize_step([img])
        f, _ = field()
        f.set_gaussians(b.get_gaussians())
        assert np.array_equal(f.render(cam).cpu().numpy(), got[k])
        f.close()
    assert np.array_equal(a.get_gaussians(), b.get_gaussians())
    a.close()
    b.close()
