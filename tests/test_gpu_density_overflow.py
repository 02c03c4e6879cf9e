"""Densities that are no numbers (a support so large that its kernel overflows FP32): every
halving of the bisection takes the lower half, as for densities that are not below the target."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iters", [1, 5, 12])
def test_ratio_of_a_density_that_is_no_number(iters):
    import paper_2101_05031_gb300 as cs
    nodes, tets = synth.kuhn_tet_mesh((2,) * 3, 4.0, 0.1, seed=3)
    grid = synth.graded_target_grid((0.0,) * 3, (8.0,) * 3, 2.0)
    got = cs.density_match(nodes, tets, grid, r_min=0.1, R=1e10, tet_n=2, vox_m=2, max_depth=0,
                           iters=iters)
    assert np.all(got["tet_ratio"] == np.float32(0.5 + 1.5 * 0.5 ** (iters + 1)))
