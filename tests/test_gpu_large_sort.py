"""Large steps (2^19 records and buffers for 3 x 2^20 instances) sort depth and tile apart; smaller ones sort
(tile, depth) keys.  On both sides of the line, for one to three tile passes, ties in depth included, the
lists are the canonical order (tile, fp32 depth bits, record) exactly, and the instance slots stay in record
order."""
import numpy as np
import pytest

import gsinputs as gi

pytestmark = pytest.mark.gpu


def _expected(ras, cams, stride):
    count, depth = ras.read(6, np.uint32).astype(np.int64), ras.read(3, np.uint32).astype(np.int64)
    rect = ras.read(5, np.uint32).reshape(-1, 2).astype(np.int64)
    gx = np.array([-(-c["width"] // 16) for c in cams])
    gy = np.array([-(-c["height"] // 16) for c in cams])
    base = np.concatenate([[0], np.cumsum(gx * gy)])
    r = np.nonzero(count)[0]
    recs = np.repeat(r, count[r])
    k = np.arange(len(recs)) - np.repeat(np.cumsum(count[r]) - count[r], count[r])
    x0, x1, y0 = rect[recs, 0] & 0xffff, rect[recs, 0] >> 16, rect[recs, 1] & 0xffff
    w, v = x1 - x0, recs // stride
    tiles = base[v] + (y0 + k // w) * gx[v] + x0 + k % w
    order = np.lexsort((recs, depth[recs], tiles))
    return recs[order], np.bincount(tiles, minlength=base[-1]), count


# (Gaussians, views, size, log-scale, takes the large path once sized): the first forward sizes the
# buffers 1.25 x and takes the general path, the next ones the path the buffers decide
@pytest.mark.parametrize("same_depth", [False, True])
@pytest.mark.parametrize("n,views,size,logscale,large", [
    (523_000, 1, (640, 480), -3.2, False), (524_288, 1, (640, 480), -3.2, True), (900_000, 1, (120, 90), -2.6, True),
    (600_000, 1, (1297, 840), -5.5, False), (600_000, 1, (1297, 840), -4.0, True), (150_000, 4, (640, 480), -3.2, True),
    (262_144, 2, (2048, 8640), -3.4, True)])
def test_lists(n, views, size, logscale, large, same_depth):
    import torch
    import paper_2503_13086_gb300 as gs
    w, h = size
    p = gi.cube_scene(n, seed=n % 97, logscale=(logscale, 0.4))
    if same_depth:
        p[2, :n] = np.random.default_rng(n).integers(0, 5, n) * 0.25 + 2.2
    cams = [gi.identity_camera(w - 16 * k, h, 0.6 * w) for k in range(views)]
    ras = gs.Raster()
    P = torch.tensor(p, device="cuda")
    for again in range(2):  # sized by the count read back, then by the buffers it left
        ras.forward(P, n, cams)
        recs, counts, count = _expected(ras, cams, p.shape[1])
        assert (views * p.shape[1] >= 1 << 19 and len(recs) * 1.25 + 1024 >= 3 << 20) == large, len(recs)
        assert np.array_equal(ras.read(9, np.uint32).astype(np.int64), recs), again
        rg = ras.read(10, np.uint32).reshape(-1, 2).astype(np.int64)
        assert np.array_equal(rg[:, 1] - rg[:, 0], counts)
        assert np.array_equal(rg[counts > 0, 0], (np.cumsum(counts) - counts)[counts > 0])
        assert np.array_equal(ras.read(7, np.uint32).astype(np.int64)[count > 0], (np.cumsum(count) - count)[count > 0])
    ras.close()


def test_nothing_in_view():
    import torch
    import paper_2503_13086_gb300 as gs
    n = 1 << 20
    P = torch.tensor(gi.cube_scene(n, seed=1, logscale=(-3.5, 0.3)), device="cuda")
    cam = gi.identity_camera(320, 200, 200.0)
    ras = gs.Raster()
    assert ras.forward(P, n, [cam])["pairs"] > 0
    P[2] *= -1.0  # all behind the camera
    out = ras.forward(P, n, [cam])
    assert out["pairs"] == 0 and not out["image"].any() and (out["T"] == 1).all()
    ras.close()


def test_autotune_grows_into_the_large_path():
    """The autotuner's sizing pass may grow the buffers past the line between two passes over the same
    views; its later passes and the steps after it agree with a session whose tiling is fixed."""
    import paper_2503_13086_gb300 as gs
    n = 600_000
    p = gi.cube_scene(n, seed=4, logscale=(-4.0, 0.3))
    cam, tgt = gi.identity_camera(1297, 840, 780.0), gi.uniform_target(1297, 840, 1)
    out = []
    for tune in (False, True):
        f = gs.Field(scene_extent=1.0, tiling=(16, 16, 256))
        f.set_gaussians(p[:, :n])
        img = f.add_image(cam, tgt)
        if tune:
            f.autotune([img], reps=2)
        losses = [f.optimize_step([img]) for _ in range(3)]
        out.append((losses, f.get_gaussians()))
        f.close()
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1])
