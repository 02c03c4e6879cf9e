"""Depth images of unusual sizes."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide", [True, False])
def test_the_longest_row_and_column(wide):
    """One row or column of 2^31 - 1 pixels (the most an image may have): its samples are
    those of a row of 4095 pixels over the same view. The long one's angles are rounded to
    2^-24 of the view, which moves a depth by 1e-6 of it but where a ray grazes."""
    import paper_2101_05031_gb300 as cs
    lat = cs.Lattice(np.array([[-2, -1, -1.5], [2, 1, 1.5]], np.float32), np.array([[0, 1]]),
                     np.array([0.3], np.float32), R=0.45)

    def view(n):
        cam = dict(eye=(0.5, 6.0, 0.4), target=(0.0, 0.0, 0.0), step=0.05)
        if wide:   # the half width of the view is tan(fov / 2) n
            return lat.render_depth(width=n, height=1, fov_y=2.0 * math.atan(0.5 / n), **cam)[0]
        return lat.render_depth(width=1, height=n, fov_y=2.0 * math.atan(0.5), **cam)[:, 0]

    n, few = 2 ** 31 - 1, 4095
    at = ((torch.arange(few, dtype=torch.float64, device="cuda") + 0.5) / few * n).long()
    got = view(n)[at].cpu().numpy()
    want = view(few).cpu().numpy()
    both = np.isfinite(got) & np.isfinite(want)
    assert both.sum() > 100 and np.isinf(want).sum() > 100
    assert (np.isfinite(got) != np.isfinite(want)).sum() <= 4   # two silhouettes
    assert (np.abs(got[both] - want[both]) > 1e-3).sum() <= 8
