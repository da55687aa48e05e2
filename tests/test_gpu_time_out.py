"""What follows a bounded wait that gave up.  The wait's kernel may leave stale words in the lists, so no kernel
after it may take an index from them: they return at once, the call reports the time-out, outputs and the
session's state stay as they were, and the next call is as if nothing had happened.  The error bit is set
by the host before the step (no wait runs out here, and no list is damaged)."""
import ctypes

import numpy as np
import pytest

import gsinputs as gi

pytestmark = pytest.mark.gpu

TIMEOUT = 6
# one step's binning in one cluster launch, by the separate kernels, and with the depth presort
SCENES = {"small": (2000, 96, 64, -3.5), "general": (60000, 640, 360, -3.5), "large": (600000, 1297, 840, -4.0)}


def _field(gs, size, seed, **kw):
    n, w, h, logscale = SCENES[size]
    f = gs.Field(scene_extent=1.0, tiling=(16, 16, 256), **kw)
    f.set_gaussians(gi.cube_scene(n, seed=seed, logscale=(logscale, 0.3))[:, :n])
    cam = gi.identity_camera(w, h, 0.6 * w)
    return f, f.add_image(cam, gi.uniform_target(w, h, seed)), cam


def _state(f):
    return list(f.get_gaussians(with_adam=True)) + [np.array([f.stats()["adam_step"], f.image_info(0, 1)[0]])]


def _times_out(gs, call):
    with pytest.raises(gs.GSError) as e:
        call()
    assert e.value.status == TIMEOUT


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("size", sorted(SCENES))
def test_session(size, use_graph):
    import paper_2503_13086_gb300 as gs
    f, img, cam = _field(gs, size, 3, use_graph=use_graph)
    twin, _, _ = _field(gs, size, 3, use_graph=use_graph)
    for steps_before in (0, 2, 1):  # the sizing step, a replayed one, the one after a render
        for _ in range(steps_before):
            assert f.optimize_step([img]) == twin.optimize_step([img])
        before = _state(f)
        for call in (lambda: f.optimize_step([img]), lambda: f.integrate(img), lambda: f.render(cam),
                     lambda: f.autotune([img], reps=1)):
            f.time_out_next()
            _times_out(gs, call)
            for a, b in zip(before, _state(f)):
                assert np.array_equal(a, b)
    assert np.array_equal(f.render(cam).cpu().numpy(), twin.render(cam).cpu().numpy())
    assert f.optimize_step([img]) == twin.optimize_step([img])
    for a, b in zip(_state(f), _state(twin)):
        assert np.array_equal(a, b)
    f.close()
    twin.close()


@pytest.mark.parametrize("size", sorted(SCENES))
def test_raster(size):
    import torch
    import paper_2503_13086_gb300 as gs
    n, w, h, logscale = SCENES[size]
    cam = gi.identity_camera(w, h, 0.6 * w)
    P = torch.tensor(gi.cube_scene(n, seed=5, logscale=(logscale, 0.3)), device="cuda")
    tgt = torch.tensor(gi.uniform_target(w, h, 5).reshape(-1), device="cuda")
    ras = gs.Raster()
    for _ in range(2):
        o = ras.forward(P, n, [cam])
    loss, d = ras.loss(o["image"], tgt)
    grads, _ = ras.backward(P, o["image"], o["last"], d)
    ras.time_out_next()
    _times_out(gs, lambda: ras.forward(P, n, [cam]))
    # without out_pairs nothing is read back: the calls that follow report it
    out = {k: torch.full_like(o[k], 7) for k in ("image", "T", "last", "gp")}
    bg = (ctypes.c_float * 3)()
    ras.time_out_next()
    p = {k: ctypes.c_void_p(v.data_ptr()) for k, v in out.items()}
    assert ras._lib.gs_raster_forward(ras._h, None, ctypes.c_void_p(P.data_ptr()), n, P.shape[1], (gs.Camera * 1)(gs.Camera.of(cam)),
                                      1, bg, p["image"], p["T"], p["last"], p["gp"], None) == 0
    torch.cuda.synchronize()
    for v in out.values():
        assert bool((v == 7).all())
    _times_out(gs, lambda: ras.loss(o["image"], tgt))
    got = torch.full_like(P, 7.0)
    assert ras._lib.gs_raster_backward(ras._h, None, ctypes.c_void_p(P.data_ptr()), p["image"], p["last"],
                                       ctypes.c_void_p(d.data_ptr()), ctypes.c_void_p(got.data_ptr()), None) == TIMEOUT
    assert bool((got == 7).all())
    again = ras.forward(P, n, [cam])
    loss2, d2 = ras.loss(again["image"], tgt)
    assert loss2 == loss and torch.equal(again["image"], o["image"])
    assert torch.equal(ras.backward(P, again["image"], again["last"], d2)[0], grads)
    ras.close()
