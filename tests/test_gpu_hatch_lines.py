"""Infill with few and many crossings per line: a warp per line up to its buffer's
size, radix sorts above it and where there are more lines than vertices. Bars with
vertical sides, so that every crossing's x is a side's x exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bars, n_lines", [(1, 3), (1, 40), (15, 9), (16, 9), (17, 12), (511, 7),
                                           (1024, 6), (1025, 6), (1024, 5000)])
def test_bars(bars, n_lines):
    import paper_2101_05031_gb300 as cs
    rng = np.random.default_rng(bars + n_lines)
    layers, sp = 3, 0.5
    xy, want, want_off = [], [], [0]
    for l in range(layers):
        k = bars if l != 1 else bars // 2               # layer 1 of a single bar: empty
        top = 0.25 + sp * min(n_lines, 6) * rng.uniform(0.3, 1.2, k)
        x = np.sort(rng.uniform(-40.0, 40.0, 2 * k).astype(np.float32)).reshape(k, 2)
        order = rng.permutation(k)
        for b in order:
            xy.append([[x[b, 0], -1.0], [x[b, 1], -1.0], [x[b, 1], top[b]], [x[b, 0], top[b]]])
        top = top.astype(np.float32)
        for m in range(n_lines):
            y = np.float32(m * sp)
            s = x[y < top]
            seg = s if m % 2 == 0 else s[::-1, ::-1]
            want += [(a, b, y) for a, b in seg]
        want_off.append(len(want))
    xy = np.asarray(xy, np.float32).reshape(-1, 2)
    lo = np.cumsum([0, bars, bars // 2, bars]).astype(np.int64)
    d = cs.DeviceContours.from_host(lo, 4 * np.arange(lo[-1] + 1, dtype=np.int64), xy)
    off, seg = d.hatch(y0=0.0, spacing=sp, n_lines=n_lines)
    assert off.tolist() == want_off
    assert np.array_equal(seg, np.asarray(want, np.float32).reshape(-1, 3))
