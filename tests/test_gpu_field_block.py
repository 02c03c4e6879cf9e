"""The block field kernel with one and two pixel rows per thread (supports below
and from 10 pixels), at grid sizes around its 8 x 8 blocks and 16 x 16 tiles, for
every slab depth, Sigma and mask, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth
from tests import helpers

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slab", [1, 2, 4, 8])
@pytest.mark.parametrize("pixel, nx, ny", [(0.05, 1, 1), (0.05, 8, 7), (0.05, 17, 33),
                                           (0.02, 31, 9), (0.02, 80, 49), (0.08, 41, 23)])
def test_rows_per_thread_against_the_oracle(slab, pixel, nx, ny):
    import paper_2101_05031_gb300 as cs
    nodes, edges, radius = synth.freudenthal(5, 1.0, 0.2, (0.15, 0.35), seed=synth.SEED_BASE + 41)
    R, nl = 0.525, 11   # 10.5, 26 and 6.6 pixels; 11 layers: a slab that is not full
    kw = dict(z0=1.31, dz=0.13, n_layers=nl, x0=1.03, y0=0.97, nx=nx, ny=ny, pixel=pixel)
    lat = cs.Lattice(nodes, edges, radius, R=R)
    sig = torch.full((nl, ny, nx), -1.0, device="cuda")
    mask = torch.full((nl, ny, (nx + 31) // 32), -1, dtype=torch.int32, device="cuda")
    lat.slice(**kw, slab=slab, field_kernel="block", contours=False, sigma_out=sig, mask_out=mask)
    got = sig.cpu().numpy()
    ref = oracle.slice_sigma(nodes, edges, radius, R=R, C=1.0, **kw)
    helpers.assert_field(got, ref, 1.0)
    words = mask.cpu().numpy().view(np.uint32)
    bits = ((words[..., None] >> np.arange(32, dtype=np.uint32)) & 1).reshape(nl, ny, -1)[..., :nx]
    assert np.array_equal(bits.astype(bool), got >= np.float32(1.0))
