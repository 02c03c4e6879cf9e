"""Step 1's targets in a mesh whose tetrahedra hold from no voxel centre to thousands, so
that lanes of one warp take their own candidates and leave theirs to a warp."""
import numpy as np
import pytest

import synth
from oracle import density as D

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cubes, power", [(1, 1.0), (4, 2.0), (5, 3.0), (6, 1.0)])
def test_targets_of_mixed_sizes(cubes, power):
    import paper_2101_05031_gb300 as cs
    nodes, tets = synth.kuhn_tet_mesh((cubes,) * 3, 4.0, 0.1, seed=31)
    side = 4.0 * cubes
    nodes = (side * (nodes / side) ** power).astype(np.float32)   # small at 0, large at the far end
    voxel = side / 23.5
    grid = synth.graded_target_grid((0.0,) * 3, (side,) * 3, voxel, period=9.0)
    r = np.random.default_rng(7)
    grid["target"] = (grid["target"] * r.uniform(0.5, 1.0, grid["target"].shape)).astype(np.float32)
    got = cs.density_match(nodes, tets, grid, r_min=0.1, tet_n=2, vox_m=2, max_depth=0, iters=7)
    assert np.array_equal(got["tets"], tets)
    want = np.array([D.tet_target(grid, nodes[t].astype(np.float64)) for t in tets])
    # 8 products and sums in FP64: below 1e-14 relative; a contained centre's is exact
    assert np.allclose(got["target"], want, rtol=1e-13, atol=0.0)
