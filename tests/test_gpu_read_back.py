"""gs_field_get_gaussians into fresh memory, memory with gaps between the rows and memory off any page
boundary: every row arrives whole and nothing between or behind the rows is written."""
import ctypes

import numpy as np
import pytest

import gsinputs as gi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 1000, 16384, 70001])
@pytest.mark.parametrize("gap", [0, 1, 5000])
def test_rows_and_gaps(n, gap):
    import paper_2503_13086_gb300 as gs
    p = gi.cube_scene(n, seed=n)
    f = gs.Field(scene_extent=1.0, tiling=(16, 16, 256))
    f.set_gaussians(p[:, :n].copy())
    stride, lead, tail = n + gap, 3, 17
    flat = np.full(lead + 59 * stride + tail, 7.5, np.float32)
    want = flat.copy()
    want[lead:lead + 59 * stride].reshape(59, stride)[:, :n] = p[:, :n]
    got_n = ctypes.c_int64()
    rc = f._lib.gs_field_get_gaussians(f._h, ctypes.c_void_p(flat.ctypes.data + 4 * lead), None, None, stride,
                                       ctypes.byref(got_n))
    assert rc == 0 and got_n.value == n
    assert np.array_equal(flat, want)
    for a in f.get_gaussians(with_adam=True)[1:]:  # fresh memory: zero moments
        assert a.shape == (59, n) and not a.any()
    f.close()
