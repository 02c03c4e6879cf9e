"""A cell whose gradient is infinite or NaN reaches the struts whose support holds one of
its samples, and no other."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 4, 8])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_nonfinite_gradient_stays_in_its_supports(m, bad):
    import paper_2101_05031_gb300 as cs
    r = np.random.default_rng(m)
    R, n = 0.3, 4000
    a = r.random((n, 3)) * 2.0
    u = r.normal(size=(n, 3))
    u[: n // 2] = np.eye(3)[r.integers(0, 3, n // 2)]   # half of them along an axis
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    b = a + u * (0.2 + r.random((n, 1)))
    nodes = np.concatenate([a, b]).astype(np.float32)
    edges = np.stack([np.arange(n), np.arange(n) + n], 1).astype(np.int32)
    radius = np.full(n, 0.02, np.float32)
    dims, h = (5, 4, 6), 0.4
    cells = dict(origin=(0.05, 0.1, 0.02), h=h, dims=dims, m=m, T=1.0)
    lat = cs.Lattice(nodes, edges, radius, R=R)
    cell = (2, 1, 3)
    g = np.zeros(dims[::-1], np.float32)
    g[cell[2], cell[1], cell[0]] = bad
    gr, gn = cs.volume_fraction_backward(lat, cells, torch.tensor(g, device="cuda"))
    gr, gn = gr.cpu().numpy(), gn.cpu().numpy()
    # distances of the cell's samples to every strut's line, and where along it
    k = (np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) / m
    p = np.array(cells["origin"]) + h * (np.array(cell) + k)
    A, B = nodes[:n].astype(np.float64), nodes[n:].astype(np.float64)
    d = B - A
    length = np.linalg.norm(d, axis=1)
    d /= length[:, None]
    q = p[:, None] - A
    t = (q * d).sum(2)
    dist = np.linalg.norm(q - t[..., None] * d, axis=2)
    margin = 1e-5   # FP32 distances of coordinates up to 3: 1e-6
    far = (dist > R + margin).all(0)
    hit = ((dist < R - margin) & (t > 0) & (t < length)).any(0)
    assert far.sum() > 1000 and hit.sum() > 100
    assert (gr[far] == 0).all() and (gn[:n][far] == 0).all() and (gn[n:][far] == 0).all()
    assert not np.isfinite(gr[hit]).any()
