"""Depth images of few pixels into many struts, for which the cells that list the struts are
larger: the same depths as in an image of more pixels with rays at the same angles."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(64, 64), (16, 32), (1, 1), (2, 64)])
def test_depths_do_not_depend_on_the_cells(size):
    import paper_2101_05031_gb300 as cs
    lat = cs.Lattice(*synth.freudenthal(60), R=0.525)
    cam = dict(eye=(95.0, -18.0, 71.0), target=(29.5, 29.5, 29.5), up=(0.0, 0.0, 1.0), fov_y=0.6,
               step=0.07, refine=20)
    w, h = size
    few = lat.render_depth(**cam, width=w, height=h).cpu().numpy()
    # odd multiples of powers of two: their centres are the same numbers in FP32
    k = int((1.5e6 / (w * h)) ** 0.5) | 1
    many = lat.render_depth(**cam, width=k * w, height=k * h).cpu().numpy()
    assert np.isfinite(few).any()
    assert np.array_equal(few, many[k // 2::k, k // 2::k])
