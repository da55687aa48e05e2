"""The depth presort of large steps works inside memory a session has anyway: the step that takes it first holds
not a byte more than the one before, and a session whose budget ends there still registers its next image."""
import numpy as np
import pytest

import gsinputs as gi

pytestmark = pytest.mark.gpu


def _field(gs, p, n, budget=0):
    f = gs.Field(scene_extent=1.0, tiling=(16, 16, 256), hbm_budget_bytes=budget)
    f.set_gaussians(p[:, :n])
    cam = gi.identity_camera(1297, 840, 780.0)
    return f, cam, f.add_image(cam, gi.uniform_target(1297, 840, 1))


@pytest.mark.parametrize("n", [524_288, 900_000])
def test_no_more_memory_than_the_general_path(n):
    import paper_2503_13086_gb300 as gs
    p = gi.cube_scene(n, seed=4, logscale=(-3.8, 0.3))
    target = gi.uniform_target(1297, 840, 2)
    f, cam, img = _field(gs, p, n)
    f.optimize_step([img])  # sized by the count read back: the general path
    general = f.stats()
    assert general["last_instances"] * 1.25 + 1024 >= 3 << 20
    f.optimize_step([img])
    large = f.stats()
    assert large["last_kernels"] != general["last_kernels"]  # the other path
    assert large["bytes_in_use"] == general["bytes_in_use"]
    f.close()
    f, cam, img = _field(gs, p, n)
    f.optimize_step([img])
    f.add_image(cam, target)
    budget = f.stats()["bytes_in_use"] + (1 << 20)
    f.close()
    f, cam, img = _field(gs, p, n, budget)
    for _ in range(2):
        f.optimize_step([img])
    other = f.add_image(cam, target)
    assert np.isfinite(f.optimize_step([other]))
    f.close()
