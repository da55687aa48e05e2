"""The blend forward's candidate walk at the list lengths where it changes shape: pairs and a lone last
candidate, whole and partial chunks of 32, one and several staged batches, pixels that stop early and
pixels outside the image.  One 16 x 16 tile, isotropic Gaussians; the reference blends the kernel's own
records front to back in float64.

Tolerance, derived: an isotropic conic's exponent terms share a sign, so its rounding is at most
4 u x 5.55 (u = 2^-24, the exponent's range is [-ln 255, 0]) = 1.3e-6; the exponential instruction adds
2^-22 and the rounding of its argument (at most 8 u ln 2), together 2.0e-6 relative on alpha.  A pixel's
transmittance carries sum alpha / (1 - alpha) <= 10 of those (it stops at 1e-4) and 2 u per factor, the
colour one more and u per sum: for 600 entries at most 11 x 2.0e-6 + 600 x 3 x 6e-8 = 1.3e-4 of the
colour scale, and the colours here are below 0.75: 1e-4.  Pixels where a decision (alpha against 1/255, T
against 1e-4) is closer than its own error are left out of the comparison of the counts."""
import numpy as np
import pytest

import gsinputs as gi
from helpers import gpu_forward

pytestmark = pytest.mark.gpu


def _scene(n, opacity, seed):
    rng = np.random.default_rng(seed)
    p = np.zeros((59, (n + 31) // 32 * 32), np.float32)
    p[0:2, :n] = rng.uniform(-1.3, 1.3, (2, n))
    p[2, :n] = rng.uniform(2.9, 3.1, n)
    p[3:6, :n] = rng.uniform(-2.2, -1.0, n)
    p[6, :n] = 1.0
    p[10, :n] = np.log(opacity / (1 - opacity))
    p[11:14, :n] = rng.uniform(-1.5, 0.8, (3, n))
    return p


def _blend64(g, w, h):
    order = g["vals"].astype(np.int64)
    m, con, rgb, op = (g["rec"][k][order].astype(np.float64) for k in ("mean2d", "conic", "rgb", "opacity"))
    py, px = np.mgrid[0:h, 0:w].astype(np.float64)
    T = np.ones((h, w))
    C = np.zeros((3, h, w))
    last, gp = np.zeros((h, w), np.int64), np.zeros((h, w), np.int64)
    neval = np.full((h, w), len(order))
    done, clear = np.zeros((h, w), bool), np.ones((h, w), bool)
    for k in range(len(order)):
        dx, dy = m[k, 0] - px, m[k, 1] - py
        power = -0.5 * (con[k, 0] * dx * dx + con[k, 2] * dy * dy) - con[k, 1] * dx * dy
        alpha = np.minimum(0.99, op[k] * np.exp(power))
        clear &= done | (np.abs(alpha * 255 - 1) > 1e-5)
        use = ~done & (power <= 0) & (alpha >= 1 / 255)
        test = T * (1 - alpha)
        clear &= ~use | (np.abs(test / 1e-4 - 1) > 1e-3)
        stop = use & (test < 1e-4)
        neval[stop] = k + 1
        done |= stop
        use &= ~stop
        C += np.where(use, alpha * T, 0.0) * rgb[k][:, None, None]
        T = np.where(use, test, T)
        last[use] = k + 1
        gp += use
    return C, T, last, gp, neval, clear


@pytest.mark.parametrize("size", [(16, 16), (13, 9)])
@pytest.mark.parametrize("opacity", [0.03, 0.9])
@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 255, 256, 257, 545])
def test_walk_edges(n, opacity, size):
    import paper_2503_13086_gb300 as gs
    w, h = size
    ras = gs.Raster()
    g = gpu_forward(ras, _scene(n, opacity, 40 + n), n, [gi.identity_camera(w, h, 16.0)])
    assert len(g["vals"]) >= 1
    C, T, last, gp, neval, clear = _blend64(g, w, h)
    out = g["out"]
    assert np.abs(out["image"].cpu().numpy().reshape(3, h, w) - C)[:, clear].max() <= 1e-4
    assert np.abs(out["T"].cpu().numpy().reshape(h, w) - T)[clear].max() <= 1.3e-4
    assert np.array_equal(out["last"].cpu().numpy().reshape(h, w)[clear], last[clear])
    assert np.array_equal(out["gp"].cpu().numpy().reshape(h, w)[clear], gp[clear])
    assert clear.mean() > 0.8
    if clear.all():
        assert out["pairs"] == int(neval.sum())
    ras.close()


def test_few_and_many_tiles_agree():
    """A picture small enough for the four-candidate walk and the same picture with a margin that takes the
    tile count past the line: the pixels both have are the same bits."""
    import torch
    import paper_2503_13086_gb300 as gs
    p = gi.cube_scene(6000, seed=9, logscale=(-3.5, 0.6))
    small = gi.identity_camera(200, 120, 150.0)
    big = dict(small, width=200 + 16 * 60, height=120 + 16 * 60)  # 13 x 8 and 73 x 68 tiles, the same origin
    # (the focal-plane clamp depends on the image size: keep it out of play)
    keep = np.abs(p[0, :6000] / p[2, :6000]) < 0.6
    p[10, :6000][~keep] = -20.0
    p[10, :6000][np.abs(p[1, :6000] / p[2, :6000]) > 0.4] = -20.0
    P = torch.tensor(p, device="cuda")
    ras = gs.Raster()
    a = ras.forward(P, 6000, [small])
    a = {k: a[k].cpu().numpy() for k in ("image", "T", "gp")}
    b = ras.forward(P, 6000, [big])
    assert np.array_equal(a["image"].reshape(3, 120, 200), b["image"].cpu().numpy().reshape(3, 1080, 1160)[:, :120, :200])
    assert np.array_equal(a["T"].reshape(120, 200), b["T"].cpu().numpy().reshape(1080, 1160)[:120, :200])
    assert np.array_equal(a["gp"].reshape(120, 200), b["gp"].cpu().numpy().reshape(1080, 1160)[:120, :200])
    ras.close()


@pytest.mark.parametrize("load", [0.0, 0.4])
@pytest.mark.parametrize("tile", [(16, 16, 256), (32, 8, 256), (16, 8, 256)])
def test_backward_item_sharing(tile, load):
    """With few (tile, chunk) items two warps share one; with many each has its own.  Both give the same
    bits: the first 40 Gaussians alone and the same 40 followed by enough others, too transparent to be
    blended, that the item count passes the line."""
    import torch
    import paper_2503_13086_gb300 as gs
    n, many = 40, 393_216
    small = _scene(n, 0.5, 7)
    big = np.zeros((59, many), np.float32)
    big[:, :n] = small[:, :n]
    big[:, n:] = small[:, :1]
    big[2, n:] = 5.0  # behind them, so that the first chunks hold the same entries
    big[10, n:] = -20.0  # opacity 2e-9: below 1/255 everywhere
    cam = gi.identity_camera(48, 33, 16.0)
    tgt = torch.tensor(gi.uniform_target(48, 33, 5).reshape(-1), device="cuda")
    got = []
    for p, k in ((small, n), (big, many)):
        ras = gs.Raster()
        ras.set_tiling(*tile)
        P = torch.tensor(p, device="cuda")
        out = ras.forward(P, k, [cam])
        _, d = ras.loss(out["image"], tgt, 0.2, lambda_load=load)
        got.append((out["image"].cpu().numpy(), ras.backward(P, out["image"], out["last"], d)[0].cpu().numpy()[:, :n]))
        ras.close()
    assert np.array_equal(got[0][0], got[1][0])
    assert np.array_equal(got[0][1], got[1][1])
    assert np.abs(got[0][1]).max() > 0
