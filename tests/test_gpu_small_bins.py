"""The small steps' binning (emission, sort, ranges and tile order in one cluster launch) and the separate
kernels beyond it, at instance counts around every change of shape: one CTA, each cluster size, one to
four keys per thread, and the last count before the separate kernels take over.  The lists are integers:
they equal the canonical order (tile, fp32 depth bits, record) exactly."""
import numpy as np
import pytest

import gsinputs as gi
from helpers import gpu_forward

pytestmark = pytest.mark.gpu


def _scene(n, seed, same_depth):
    p = gi.cube_scene(n, seed=seed, stride=(n + 31) // 32 * 32, logscale=(-6.0, 0.3))
    if same_depth:  # ties: the record index decides
        p[2, :n] = np.random.default_rng(seed).integers(0, 3, n) * 0.25 + 2.5
    return p


def _expected(ras, g, cams, stride):
    """Instances by record, then the canonical stable order."""
    rect = ras.read(5, np.uint32).reshape(-1, 2)
    gx = [-(-c["width"] // 16) for c in cams]
    gy = [-(-c["height"] // 16) for c in cams]
    base = np.concatenate([[0], np.cumsum([a * b for a, b in zip(gx, gy)])])
    tiles, recs = [], []
    for r in np.nonzero(g["count"])[0]:
        x0, x1, y0, y1 = rect[r, 0] & 0xffff, rect[r, 0] >> 16, rect[r, 1] & 0xffff, rect[r, 1] >> 16
        v = r // stride
        for y in range(y0, y1):
            for x in range(x0, x1):
                tiles.append(base[v] + y * gx[v] + x)
                recs.append(r)
    tiles, recs = np.array(tiles, np.int64), np.array(recs, np.int64)
    depth = g["depth"].view(np.uint32)[recs].astype(np.int64)
    order = np.lexsort((recs, depth, tiles))
    counts = np.bincount(tiles, minlength=base[-1])
    return recs[order], counts


# Gaussians of about one and a half tiles each; the raster's capacity is 1.25 x the instances + 1024
@pytest.mark.parametrize("same_depth", [False, True])
@pytest.mark.parametrize("views", [1, 3])
@pytest.mark.parametrize("n", [1, 3, 700, 1500, 3000, 5000, 11000, 24000, 36000])
def test_lists(n, views, same_depth):
    import paper_2503_13086_gb300 as gs
    if views == 3:
        n = (n + 2) // 3
    cams = [gi.identity_camera(w, h, 200.0) for w, h in [(250, 190), (131, 77), (64, 300)][:views]]
    ras = gs.Raster()
    p = _scene(n, 3 + n, same_depth)
    g = gpu_forward(ras, p, n, cams)
    recs, counts = _expected(ras, g, cams, p.shape[1])
    assert np.array_equal(g["vals"].astype(np.int64), recs)
    L = (g["ranges"][:, 1] - g["ranges"][:, 0]).astype(np.int64)
    assert np.array_equal(L, counts)
    starts = np.concatenate([[0], np.cumsum(counts)[:-1]])
    assert np.array_equal(g["ranges"][:, 0][counts > 0].astype(np.int64), starts[counts > 0])
    ras.close()


def test_both_sides_of_the_line_agree():
    """The same step binned by the cluster and, with instance buffers grown by an earlier larger step, by
    the separate kernels: the same image and gradient bits."""
    import torch
    import paper_2503_13086_gb300 as gs
    n = 4000
    p = _scene(n, 5, False)
    cam = gi.identity_camera(250, 190, 200.0)
    tgt = torch.tensor(gi.uniform_target(250, 190, 1).reshape(-1), device="cuda")
    big = torch.tensor(gi.cube_scene(40000, seed=2, stride=40000, logscale=(-3.0, 0.3)), device="cuda")
    got = []
    for grow in (False, True):
        ras = gs.Raster()
        if grow:
            ras.forward(big, 40000, [cam])
        P = torch.tensor(p, device="cuda")
        o = ras.forward(P, n, [cam])
        _, d = ras.loss(o["image"], tgt, 0.2)
        got.append((o["image"].cpu().numpy(), o["last"].cpu().numpy(), o["pairs"],
                    ras.backward(P, o["image"], o["last"], d)[0].cpu().numpy(), ras.read(9, np.uint32)))
        ras.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
