"""Long loops by the number of their splitters, counted here with the sampling that cuts them:
in one block with up to 196 KB of links, just below and just above what it takes, and with too
many to go ahead of their count; and each loop's area against its pixels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BLOCK, AHEAD = 12288, 1 << 17


@pytest.mark.parametrize("bars, length, low, high", [(16, 40.0, 3073, 8192), (48, 40.0, 12000, BLOCK),
                                                     (49, 40.0, BLOCK + 1, 12500),
                                                     (730, 60.0, AHEAD + 1, 150000)])
def test_long_loops(bars, length, low, high):
    import paper_2101_05031_gb300 as cs
    px = 0.02
    y = 0.2 * np.arange(bars) + 0.3
    nodes = np.concatenate([np.stack([np.full(bars, x), y, np.zeros(bars)], 1)
                            for x in (0.5, 0.5 + length)]).astype(np.float32)
    edges = np.stack([np.arange(bars), np.arange(bars) + bars], 1).astype(np.int32)
    lat = cs.Lattice(nodes, edges, np.full(bars, 0.05, np.float32), R=0.075)
    nx, ny = int((length + 1.0) / px), int((y[-1] + 0.3) / px)
    mask = torch.zeros((1, ny, (nx + 31) // 32), dtype=torch.int32, device="cuda")
    c = lat.slice(z0=0.0, dz=0.1, n_layers=1, x0=0.0, y0=0.0, nx=nx, ny=ny, pixel=px,
                  edge_ids=True, mask_out=mask)
    words = mask.cpu().numpy().view(np.uint32)[0]
    inside = ((words[..., None] >> np.arange(32, dtype=np.uint32)) & 1).reshape(ny, -1)[:, :nx]
    pad = np.zeros((ny + 2, nx + 2), bool)
    pad[1:-1, 1:-1] = inside
    W = nx + 2
    J, I = np.nonzero(pad[:, :-1] != pad[:, 1:])
    K, L = np.nonzero(pad[:-1] != pad[1:])
    want = np.sort(np.concatenate([2 * (J * W + I), 2 * (K * W + L) + 1]))
    assert np.array_equal(np.sort(c.edge_id), want)   # every crossing once
    n = len(want)
    # splitters: one crossing in 8 (16, 32) by a hash of its number, and the local minima
    bits = 3 if n <= 1 << 16 else (4 if n <= 1 << 18 else 5)
    sampled = int(((np.arange(n, dtype=np.uint32) * np.uint32(2654435761))
                   >> np.uint32(32 - bits) == 0).sum())
    assert low <= sampled and sampled + 2 * bars <= high
    off = c.loop_vert_off
    assert len(off) == bars + 1 and c.layer_loop_off.tolist() == [0, bars]
    heads = c.edge_id[off[:-1]]
    assert np.all(np.diff(heads) > 0)                 # loops listed by their heads
    assert np.array_equal(heads, np.minimum.reduceat(c.edge_id, off[:-1]))
    rows = np.add.reduceat(inside.sum(1), np.concatenate([[0], ((y[1:] - 0.1) / px).astype(int)]))
    for b in range(bars):
        p = c.xy[off[b]:off[b + 1]].astype(np.float64)
        q = np.roll(p, -1, 0)
        assert np.max(np.abs(q - p)) < 1.5 * px       # on edges of one cell
        area = 0.5 * np.sum(p[:, 0] * q[:, 1] - q[:, 0] * p[:, 1]) / px ** 2
        assert abs(area - rows[b]) <= 0.5 * len(p)    # half a pixel along the boundary
