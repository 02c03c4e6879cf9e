"""A bounded wait of the field kernel that gave up is reported by every call that
evaluates the field, once."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELLS = dict(origin=(0.0, 0.0, 0.0), h=0.5, dims=(2, 2, 2), m=4, T=0.05)


def _forward(cs, lat):
    return cs.volume_fraction(lat, CELLS)


def _backward(cs, lat):
    return cs.volume_fraction_backward(lat, CELLS, torch.ones((2, 2, 2), device="cuda"))[0]


def _slice(cs, lat):
    out = torch.empty((2, 16, 16), device="cuda")
    lat.slice(z0=0.2, dz=0.1, n_layers=2, x0=0.0, y0=0.0, nx=16, ny=16, pixel=0.06,
              contours=False, sigma_out=out)
    return out


@pytest.mark.parametrize("call", [_forward, _backward, _slice])
def test_timeout_reaches_the_caller_once(call):
    import paper_2101_05031_gb300 as cs
    lat = cs.Lattice(np.array([[0.1, 0.2, 0.1], [0.8, 0.7, 0.9]], np.float32), np.array([[0, 1]]),
                     np.array([0.2], np.float32), R=0.3)
    want = call(cs, lat).clone()
    assert cs.load().csl_debug_lattice_timeout(lat.handle, 1000, None) == 0
    with pytest.raises(cs.CslError) as e:
        call(cs, lat)
    assert e.value.code == 4
    assert torch.equal(call(cs, lat), want)   # the next call is healthy
