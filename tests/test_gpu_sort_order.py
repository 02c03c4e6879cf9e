"""The stable radix sort by itself: every pair where numpy's stable sort puts it, at one tile,
around whole tiles and with a ragged last one."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 2, 33, 255, 4095, 4096, 4097, 8191, 8192, 12289, 70001])
@pytest.mark.parametrize("bits, kinds", [(1, 2), (8, 1), (8, 256), (9, 7), (16, 300), (17, 1 << 17),
                                         (32, 1 << 32)])
def test_every_pair_in_its_place(n, bits, kinds):
    import paper_2101_05031_gb300 as cs
    r = np.random.default_rng(n + bits)
    # kinds different keys, the largest of `bits` bits among them
    keys = ((1 << bits) - 1 - r.integers(0, kinds, n)).astype(np.uint32)
    vals = r.permutation(n).astype(np.uint32)
    k = torch.tensor(keys.view(np.int32), device="cuda")
    v = torch.tensor(vals.view(np.int32), device="cuda")
    k0, v0 = (t if n else torch.zeros(1, dtype=torch.int32, device="cuda") for t in (k, v))
    lib = cs.load()
    assert lib.csl_debug_sort_pairs(ctypes.c_void_p(k0.data_ptr()), ctypes.c_void_p(v0.data_ptr()), n,
                                    bits, None) == 0
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(k.cpu().numpy().view(np.uint32), keys[order])
    assert np.array_equal(v.cpu().numpy().view(np.uint32), vals[order])
