"""Simplification, smoothing and infill where loops meet the 1024-vertex spans
their kernels work on: loops that end, start and straddle at span edges, loops
longer than several spans, runs of empty loops, and counts not divisible by 4."""
import numpy as np
import pytest

from oracle import simplify as Z

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _squares(sizes, layers, nx, seed):
    """Loops with the given vertex counts (0: an empty loop), each vertex on a
    grid edge of its own in its layer, near a line so that some are dropped."""
    r = np.random.default_rng(seed)
    W = nx + 2
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    xy = np.zeros((off[-1], 2), np.float32)
    eid = np.zeros(off[-1], np.int32)
    per = -(-len(sizes) // layers)
    lo = np.minimum(np.arange(layers + 1) * per, len(sizes)).astype(np.int64)
    for k in range(layers):
        v0, v1 = off[lo[k]], off[lo[k + 1]]
        n = v1 - v0
        # every third sample's horizontal edge, row by row: neighbours in a loop
        # lie three cells apart, so no cell has two crossings
        s = 3 * np.arange(n)
        assert 3 * n < W * W
        eid[v0:v1] = 2 * s
        xy[v0:v1, 0] = 0.01 * (s % W) + 0.004 * r.random(n)
        xy[v0:v1, 1] = 0.01 * (s // W)
    return lo, off, xy, eid


SIZES = {
    "span_edges": [1000, 24, 1024, 5, 4, 3, 1012, 1, 1023, 7],
    "straddling": [37] * 150 + [1025, 6],
    "long": [5000, 3, 9, 2049],
    "empty_runs": [0, 0, 1024, 0, 0, 0, 5] + [0] * 1500 + [11, 0, 1013, 0],
    "tiny": [3],
}


@pytest.mark.parametrize("name", sorted(SIZES))
def test_simplify_at_span_edges(name):
    import paper_2101_05031_gb300 as cs
    nx, tol = 180, 0.0015
    lo, off, xy, eid = _squares(SIZES[name], 2 if len(SIZES[name]) > 3 else 1, nx, 5)
    dev = cs.DeviceContours.from_host(lo, off, xy, eid)
    got = dev.simplify(nx, nx, tol).to_host()
    assert np.array_equal(got.layer_loop_off, lo)
    dropped = 0
    for k in range(len(lo) - 1):
        v0, v1 = off[lo[k]], off[lo[k + 1]]
        roff, reid, rxy, _ = Z.simplify_layer(off[lo[k]:lo[k + 1] + 1] - v0, eid[v0:v1], xy[v0:v1],
                                              nx, tol)
        goff = got.loop_vert_off[lo[k]:lo[k + 1] + 1]
        assert np.array_equal(goff - goff[0], roff)
        assert np.array_equal(got.edge_id[goff[0]:goff[-1]], reid)
        assert np.array_equal(got.xy[goff[0]:goff[-1]], rxy)
        dropped += (v1 - v0) - len(reid)
    assert dropped > 0 or name == "tiny"


@pytest.mark.parametrize("name", sorted(SIZES))
def test_smooth_at_span_edges(name):
    """One step moves each vertex toward its own loop's neighbours only."""
    import paper_2101_05031_gb300 as cs
    nx, px = 180, np.float32(0.01)
    lo, off, xy, eid = _squares(SIZES[name], 2 if len(SIZES[name]) > 3 else 1, nx, 6)
    dev = cs.DeviceContours.from_host(lo, off, xy, eid)
    got = dev.smooth(0.005, 0.005, float(px), nx, nx, lam=0.5, margin=0.05, iterations=1).to_host()
    want = xy.copy()
    I = (eid // 2) % (nx + 2)
    low = np.float32(0.005 - 0.5 * 0.01) + I.astype(np.float32) * px
    b0, b1 = low + np.float32(0.05 * 0.01), low + np.float32((1 - 0.05) * 0.01)
    for a, b in zip(off[:-1], off[1:]):
        if b - a < 3:
            continue
        x = xy[a:b, 0]
        m = np.float32(0.5) * (np.roll(x, 1) + np.roll(x, -1))
        want[a:b, 0] = np.minimum(np.maximum(x + np.float32(0.5) * (m - x), b0[a:b]), b1[a:b])
    assert np.array_equal(got.xy, want)
