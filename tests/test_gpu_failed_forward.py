"""After a forward that failed (a bad camera, more instances than a list can hold) there is nothing for a loss,
a backward or a read: they are refused, and the next forward works as on a rasterizer of its own."""
import numpy as np
import pytest

import gsinputs as gi

pytestmark = pytest.mark.gpu

STATE, INVALID, CAPACITY = 7, 1, 4


@pytest.mark.parametrize("why", ["camera", "instances"])
def test_nothing_to_go_on(why):
    import torch
    import paper_2503_13086_gb300 as gs
    n, w, h = 3000, 320, 200
    cam = gi.identity_camera(w, h, 300.0)
    P = torch.tensor(gi.cube_scene(n, seed=1), device="cuda")
    tgt = torch.tensor(gi.uniform_target(w, h, 1).reshape(-1), device="cuda")
    ras = gs.Raster()
    for _ in range(2):  # the second one is enqueued at the first one's sizes
        o = ras.forward(P, n, [cam])
    loss, d = ras.loss(o["image"], tgt)
    g, _ = ras.backward(P, o["image"], o["last"], d)
    if why == "camera":
        bad, expect = lambda: ras.forward(P, n, [dict(cam, fx=-1.0)]), INVALID
    else:  # a million Gaussians over all 2200 tiles
        m = 1 << 20
        q = np.zeros((59, m), np.float32)
        q[2], q[3:6], q[6] = 3.0, 3.0, 1.0
        Q = torch.tensor(q, device="cuda")
        bad, expect = lambda: ras.forward(Q, m, [gi.identity_camera(800, 704, 700.0)]), CAPACITY
    with pytest.raises(gs.GSError) as e:
        bad()
    assert e.value.status == expect
    for call in (lambda: ras.loss(o["image"], tgt), lambda: ras.backward(P, o["image"], o["last"], d),
                 lambda: ras.read(6, np.uint32)):
        with pytest.raises(gs.GSError) as e:
            call()
        assert e.value.status == STATE
    o2 = ras.forward(P, n, [cam])
    loss2, d2 = ras.loss(o2["image"], tgt)
    assert loss2 == loss and torch.equal(o2["image"], o["image"])
    assert torch.equal(ras.backward(P, o2["image"], o2["last"], d2)[0], g)
    ras.close()
