"""Contour emission where it can go wrong: rows of more than one segment of 1024
samples and of more than one list of crossings, bands that end inside a block, saddles
on the seams of words and segments. The contours of the field kernels are compared
with marching squares on the host over the same field and mask."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _loops(sig, C, x0, y0, px):
    """Loops of one layer: per loop (by smallest edge id) its edge ids and vertices."""
    ny, nx = sig.shape
    W = nx + 2
    S = np.zeros((ny + 2, W), np.float32)
    S[1:-1, 1:-1] = sig
    inside = np.zeros(S.shape, bool)
    inside[1:-1, 1:-1] = sig >= np.float32(C)
    side_edge = (lambda J, I: 2 * (J * W + I), lambda J, I: 2 * (J * W + I + 1) + 1,
                 lambda J, I: 2 * ((J + 1) * W + I), lambda J, I: 2 * (J * W + I) + 1)
    c = np.stack([inside[:-1, :-1], inside[:-1, 1:], inside[1:, 1:], inside[1:, :-1]])
    succ = {}
    for J, I in np.argwhere(c.any(0) & ~c.all(0)):
        s = c[:, J, I]
        ent = [k for k in range(4) if s[k] and not s[(k + 1) & 3]]
        lea = [k for k in range(4) if not s[k] and s[(k + 1) & 3]]
        if len(ent) == 1:
            succ[side_edge[ent[0]](J, I)] = side_edge[lea[0]](J, I)
        else:
            w = np.float32(0.25) * (((S[J, I] + S[J, I + 1]) + S[J + 1, I + 1]) + S[J + 1, I])
            for k in ent:
                succ[side_edge[k](J, I)] = side_edge[(k + (1 if w >= np.float32(C) else 3)) & 3](J, I)
    loops, seen = [], set()
    for h in sorted(succ):
        if h in seen:
            continue
        ids, e = [], h
        while e not in seen:
            seen.add(e)
            ids.append(e)
            e = succ[e]
        loops.append(ids)
    eid = np.concatenate([np.array(q) for q in loops])
    J, I, d = (eid >> 1) // W, (eid >> 1) % W, eid & 1
    v0, v1 = S[J, I].astype(np.float64), S[J + d, I + 1 - d].astype(np.float64)
    t = (np.float64(np.float32(C)) - v0) / (v1 - v0)
    x = x0 + (I - 0.5 + np.where(d == 0, t, 0.0)) * px
    y = y0 + (J - 0.5 + np.where(d == 1, t, 0.0)) * px
    return np.cumsum([0] + [len(q) for q in loops]), eid, np.stack([x, y], 1)


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("nx,ny,pitch", [(1021, 17, 2.3), (1022, 15, 2.3), (1024, 33, 3.1),
                                         (2055, 14, 2.3), (31, 31, 2.3), (1, 1, 2.0), (33, 16, 9.0)])
def test_dense_rows(nx, ny, pitch, fused):
    import paper_2101_05031_gb300 as cs
    rng = np.random.default_rng(nx * 64 + ny)
    px = 0.1
    gx, gy = np.meshgrid(np.arange(0, nx + pitch, pitch), np.arange(0, ny + pitch, pitch))
    p = np.stack([gx.ravel(), gy.ravel()], 1) + rng.uniform(-0.4, 0.4, (gx.size, 2))
    p *= px
    k = len(p)
    nodes = np.zeros((2 * k, 3), np.float32)
    nodes[:k, :2] = p
    nodes[k:, :2] = p + rng.uniform(-0.03, 0.03, (k, 2))
    nodes[:k, 2], nodes[k:, 2] = -0.5, 0.7
    edges = np.stack([np.arange(k), np.arange(k) + k], 1).astype(np.int32)
    r = rng.uniform(0.08, 0.13, k).astype(np.float32)
    lat = cs.Lattice(nodes, edges, r, R=1.5 * float(r.max()))
    win = dict(z0=0.0, dz=0.11, n_layers=3, x0=px / 2, y0=px / 2, nx=nx, ny=ny, pixel=px)
    cont = lat.slice(**win, edge_ids=True, fused=fused)
    sig = torch.empty(3, ny, nx, dtype=torch.float32, device="cuda")
    lat.slice(**win, sigma_out=sig, contours=False)
    sig = sig.cpu().numpy()
    for l in range(3):
        off, eid, xy = _loops(sig[l], lat.C, win["x0"], win["y0"], px)
        a, b = cont.layer_loop_off[l], cont.layer_loop_off[l + 1]
        lo = np.asarray(cont.loop_vert_off[a:b + 1])
        assert np.array_equal(lo - lo[0], off)
        assert np.array_equal(cont.edge_id[lo[0]:lo[-1]], eid)
        # in pixels: t <= 1 to two differences, a division (2 ulp) and a rounding, then
        # four roundings of a coordinate of up to n + 2 pixels; twice that
        tol = px * (1e-6 + 2 ** -23 * 4 * (max(nx, ny) + 2))
        assert np.abs(cont.xy[lo[0]:lo[-1]] - xy).max() <= tol
