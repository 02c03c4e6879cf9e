"""The stable radix sort at one tile, just above it and with a ragged last tile,
through what orders by it: records by lower z with equal keys in input order."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 255, 4095, 4096, 4097, 8192, 12289, 70001])
@pytest.mark.parametrize("levels", [1, 7, 100000])
def test_stable_order_of_records(n, levels):
    """One tile of pixels with every strut in it: the list is the sort's output, the
    strut ids in order of (lower z, id)."""
    import paper_2101_05031_gb300 as cs
    r = np.random.default_rng(n + levels)
    z = (r.integers(0, levels, n) * (0.9 / levels)).astype(np.float32)
    nodes = np.zeros((2 * n, 3), np.float32)
    nodes[0::2, 2] = z
    nodes[1::2, 2] = z + np.float32(0.05)
    nodes[:, :2] = 0.5 + 0.1 * r.random((2 * n, 2))
    edges = np.arange(2 * n, dtype=np.int32).reshape(-1, 2)
    lat = cs.Lattice(nodes, edges, np.full(n, 0.01, np.float32), R=0.02)
    sigma = torch.empty((1, 16, 16), device="cuda")
    lat.slice(z0=0.5, dz=1.0, n_layers=1, x0=0.0, y0=0.0, nx=16, ny=16, pixel=0.07,
              contours=False, sigma_out=sigma)
    # host-resident preparation sorts in batches and merges: the same records, so the
    # same sums in the same order, bit for bit
    out = cs.Lattice(nodes, edges, np.full(n, 0.01, np.float32), R=0.02, host_resident=True,
                     batch_edges=max(1, n // 3))
    other = torch.empty_like(sigma)
    out.slice(z0=0.5, dz=1.0, n_layers=1, x0=0.0, y0=0.0, nx=16, ny=16, pixel=0.07,
              contours=False, sigma_out=other)
    assert torch.equal(sigma, other)
    off, ids = lat.slab_bins(z0=0.5, dz=1.0, first_layer=0, n_slab_layers=1, x0=0.0, y0=0.0,
                             nx=16, ny=16, pixel=0.07)
    want = np.nonzero((z - np.float32(0.0199) <= 0.5) & (z + np.float32(0.0699) >= 0.5))[0]
    assert set(want) <= set(ids.tolist()) and len(set(ids.tolist())) == len(ids)
