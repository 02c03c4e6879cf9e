"""Loop assembly where loops are long (many splitters each): resolved by one
block, just above what a block takes, and with too many splitters to go ahead of
the count; the loops checked against the binary image alone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bars, length", [(3, 40.0), (60, 40.0), (140, 40.0), (700, 60.0)])
def test_long_loops(bars, length):
    """Bars along x in one plane, each a contour of about 2 length / pixel vertices:
    about 400, 7,500, 17,500 and 130,000 splitters in long cycles."""
    import paper_2101_05031_gb300 as cs
    px, rho, R = 0.02, 0.05, 0.075
    y = 0.2 * np.arange(bars) + 0.3
    nodes = np.concatenate([np.stack([np.full(bars, x), y, np.zeros(bars)], 1)
                            for x in (0.5, 0.5 + length)]).astype(np.float32)
    edges = np.stack([np.arange(bars), np.arange(bars) + bars], 1).astype(np.int32)
    lat = cs.Lattice(nodes, edges, np.full(bars, rho, np.float32), R=R)
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
    off = c.loop_vert_off
    assert len(off) == bars + 1 and c.layer_loop_off.tolist() == [0, bars]
    heads = c.edge_id[off[:-1]]
    assert np.all(np.diff(heads) > 0)                 # loops listed by their heads
    assert np.array_equal(heads, np.minimum.reduceat(c.edge_id, off[:-1]))
    # consecutive vertices (the last and the first too) lie on edges of one cell: less
    # than 1.5 pixels apart, and the area is the inside pixels' within half a boundary
    for a, b in zip(off[:-1], off[1:]):
        p = c.xy[a:b].astype(np.float64)
        q = np.roll(p, -1, 0)
        assert np.max(np.abs(q - p)) < 1.5 * px
        area = 0.5 * np.sum(p[:, 0] * q[:, 1] - q[:, 0] * p[:, 1])
        assert area > 0.0                             # inside on the left
