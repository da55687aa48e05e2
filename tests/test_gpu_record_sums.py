"""The per-record sums of the instance gradients (K9a): records inside one 32-instance chunk, over a few
chunks (added by their own thread) and over many (added by their warp, in batches of 32 chunks), next to
one another as an arrival's large Gaussians are.  Reference: the kernel's own instance gradients summed in
float64; a float32 sum of c terms in any order is within c u sum |x| of it (u = 2^-24)."""
import numpy as np
import pytest

import gsinputs as gi

pytestmark = pytest.mark.gpu


# tiles across the image: 2 x 2 (inside a chunk) up to 90 x 60 (169 chunks, six batches)
@pytest.mark.parametrize("views", [1, 2])
@pytest.mark.parametrize("size", [(32, 32), (160, 160), (200, 176), (512, 512), (544, 528), (1440, 960)])
def test_sums(size, views):
    import torch
    import paper_2503_13086_gb300 as gs
    w, h = size
    n, large = 300, 70
    p = gi.cube_scene(n, seed=w, stride=320, logscale=(-3.0, 0.3))
    p[3:6, 100:100 + large] = 1.5  # these cover the image
    p[0:2, 100:100 + large] *= 0.1
    p[10, 100:100 + large] = -4.0
    cams = [gi.identity_camera(w, h, 0.9 * w) for _ in range(views)]
    ras = gs.Raster()
    P = torch.tensor(p, device="cuda")
    out = ras.forward(P, n, cams)
    d = torch.randn(out["image"].shape, generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    _, g2 = ras.backward(P, out["image"], out["last"], d, want_grad2d=True)
    count, off = ras.read(6, np.uint32).astype(np.int64), ras.read(7, np.uint32).astype(np.int64)
    inst = ras.read(12, np.float32).reshape(-1, 12)[:, :9].astype(np.float64)
    got = g2.cpu().numpy().reshape(-1, 9).astype(np.float64)
    assert count.max() >= min(4, (w // 16) * (h // 16))
    for r in np.nonzero(count)[0]:
        x = inst[off[r]:off[r] + count[r]]
        bound = count[r] * 2.0 ** -24 * np.abs(x).sum(0)
        assert (np.abs(got[r] - x.sum(0)) <= bound + 1e-30).all(), (r, count[r])
    ras.close()
