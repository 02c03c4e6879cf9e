"""Infill of rows of bars whose neighbours cross the same lines: short and long lines, sides
of more lines than a warp has lanes, and so many vertices per line that each line has several
counters. Vertical sides, so that every crossing's x is a side's x exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rows(per_row, rows, height):
    """Lower left corners, widths and heights of bars in rows, as slicing lists them."""
    j, i = np.divmod(np.arange(per_row * rows), per_row)
    return np.stack([i * 1.0, j * 1.0 + 0.01 * (i % 7), np.full(i.size, 0.5), height + 0.02 * (i % 5)], 1)


@pytest.mark.parametrize("parts, n_lines, sp", [
    ([_rows(70, 50, 0.6)] * 2, 200, 0.3),             # lines of 140 crossings
    ([_rows(1200, 3, 0.6), _rows(30, 9, 0.6)], 12, 0.3),   # one line in four too long for a warp
    ([np.concatenate([_rows(300, 20, 0.6), _rows(5, 1, 33.0) - [7.5, 0, 0, 0]])] * 2, 500, 0.07),
    ([_rows(1100, 1, 30.0)], 90, 0.31),               # long lines, sides of 97 lines
    ([_rows(9000, 1, 0.6)], 1, 0.3),                  # 36,000 vertices for one line
    ([_rows(500, 4, 0.6)] * 3, 13, 0.045),            # sides of 13 lines, 16 counters per line
    ([_rows(400, 1, 2.0)] * 2, 48, 0.04),             # sides of 48 lines by their own lanes
    # sides of 1024, 1025, 2049 and 3,300 lines beside short ones; in lines too long for a warp
    ([np.concatenate([_rows(40, 60, 0.6), [[-2, 0, 0.5, 30.705], [-4, 0, 0.5, 30.735],
                                           [-6, 3, 0.5, 61.455], [-8, 0, 0.5, 99.0]]])] * 2, 3400, 0.03),
    ([np.concatenate([_rows(1100, 1, 30.0), [[-2, 0.0, 0.5, 12.0]]])], 1300, 0.02),
    ([_rows(40, 30, 0.6), _rows(1, 1, 0.6)[:0], _rows(1, 1, 31.0)], 100, 0.3),   # an empty layer
])
def test_rows(parts, n_lines, sp):
    import paper_2101_05031_gb300 as cs
    xy, want, want_off = [], [], [0]
    ys = (np.arange(n_lines) * sp).astype(np.float32)
    for bars in parts:
        x0, x1 = bars[:, 0].astype(np.float32), (bars[:, 0] + bars[:, 2]).astype(np.float32)
        y0, y1 = bars[:, 1].astype(np.float32), (bars[:, 1] + bars[:, 3]).astype(np.float32)
        xy.append(np.stack([np.stack(p, 1) for p in ((x0, y0), (x1, y0), (x1, y1), (x0, y1))], 1))
        for m, y in enumerate(ys):
            on = (y0 <= y) & (y < y1)
            s = np.stack([x0[on], x1[on]], 1)
            s = s[np.argsort(s[:, 0])]
            want.append(np.concatenate([s if m % 2 == 0 else s[::-1, ::-1],
                                        np.full((len(s), 1), y, np.float32)], 1))
        want_off.append(sum(len(w) for w in want))
    loops = np.cumsum([0] + [len(b) for b in parts])
    d = cs.DeviceContours.from_host(loops, 4 * np.arange(loops[-1] + 1),
                                    np.concatenate(xy).reshape(-1, 2))
    for _ in range(2):   # the slots come from atomics: the order must not show
        off, seg = d.hatch(y0=0.0, spacing=sp, n_lines=n_lines)
        assert off.tolist() == want_off
        assert np.array_equal(seg, np.concatenate(want))
