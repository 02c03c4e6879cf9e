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


@pytest.mark.parametrize("size", [(1, 1), (1, 50), (50, 1), (2, 33), (33, 2), (3, 40), (40, 3),
                                  (4, 129), (129, 4), (5, 31), (31, 5), (7, 3), (8, 4), (9, 5),
                                  (17, 9)])
def test_narrow_images(size):
    """Images narrower or lower than a warp's 8 x 4 pixels and just above them, every pixel
    against the oracle."""
    import paper_2101_05031_gb300 as cs
    import synth
    from oracle import render as V
    cfg = synth.config(1)
    lat = cs.Lattice(cfg["nodes"], cfg["edges"], cfg["radius"], R=cfg["R"])
    cam = dict(eye=(31.0, -17.0, 24.0), target=(10.0, 10.0, 9.0), up=(0.0, 0.0, 1.0),
               fov_y=0.9 / max(1.0, size[0] / size[1]), width=size[0], height=size[1])
    out = torch.full((size[1] + 2, size[0]), -1.0, device="cuda")   # rows of its neighbours
    lat.render_depth(**cam, step=0.05, refine=20, out=out[1:-1])
    out = out.cpu().numpy()
    assert (out[[0, -1]] == -1.0).all()
    ref = V.render(cfg["nodes"], cfg["edges"], cfg["radius"], R=cfg["R"], C=1.0, step=0.05,
                   refine=20, **cam)
    # as for the larger images: FP32 positions of about 40 mm; a grazing ray or a sample at
    # C within rounding can decide the other way
    bad = sum(not (np.isinf(t) and np.isinf(out[j + 1, i])) and not abs(out[j + 1, i] - t) <= 2e-3
              for (j, i), t in ref.items())
    assert bad <= 0.01 * len(ref) + 1, bad


@pytest.mark.parametrize("kind", ["any", "along an axis", "in a plane", "nearly in a plane", "short"])
@pytest.mark.parametrize("shift", [0.0, 300.0])
def test_struts_across_many_cells(kind, shift):
    """Struts up to 150 cells long, in every direction, and of no length: the cells they are
    listed in, so the image, against the oracle."""
    import paper_2101_05031_gb300 as cs
    from oracle import render as V
    r = np.random.default_rng(len(kind))
    n, R, rho = 14, 0.3, 0.22
    a = r.random((n, 3)) * 30.0
    d = r.normal(size=(n, 3))
    if kind == "along an axis":
        d = np.eye(3)[np.arange(n) % 3] * 1.0
    elif kind != "any":
        d[np.arange(n), np.arange(n) % 3] *= 0.0 if kind == "in a plane" else 1e-5
    length = 20.0 + 10.0 * r.random(n)
    if kind == "short":
        length = np.where(np.arange(n) % 5, 3.0, 0.0)
    b = a + d / np.linalg.norm(d, axis=1, keepdims=True) * length[:, None]
    nodes = (np.concatenate([a, b]) + shift).astype(np.float32)
    edges = np.stack([np.arange(n), np.arange(n) + n], 1).astype(np.int32)
    radius = np.full(n, rho, np.float32)
    lat = cs.Lattice(nodes, edges, radius, R=R)
    c = 15.0 + shift
    cam = dict(eye=(c + 60.0, c - 45.0, c + 35.0), target=(c, c, c), up=(0.0, 0.0, 1.0), fov_y=0.5,
               width=40, height=30, step=0.1, refine=20)
    depth = lat.render_depth(**cam).cpu().numpy()
    ref = V.render(nodes, edges, radius, R=R, C=1.0, **cam)
    # FP32 positions: 8 ulp of the eye's coordinates (2e-4 at 400 mm) over the sine of the
    # incidence; a ray that grazes can decide the other way
    hits = sum(np.isfinite(t) for t in ref.values())
    bad = sum(not (np.isinf(t) and np.isinf(depth[p])) and not abs(depth[p] - t) <= 5e-3
              for p, t in ref.items())
    assert hits > (5 if kind == "short" else 40)
    assert bad <= 0.02 * len(ref), bad
