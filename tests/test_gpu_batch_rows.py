"""Batches whose supports reach 10 pixels (two pixel rows per thread) in all jobs, in some and
in none, at every number of CTAs per SM: the same field and contours as job by job, and the
number that is reported is one that fits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _lattice(cs, seed):
    r = np.random.default_rng(seed)
    n = 150
    a = r.random((n, 3)) * [6.0, 5.0, 3.0]
    b = a + r.normal(size=(n, 3)) * 0.8
    return cs.Lattice(np.concatenate([a, b]).astype(np.float32),
                      np.stack([np.arange(n), np.arange(n) + n], 1).astype(np.int32),
                      r.uniform(0.1, 0.2, n).astype(np.float32), R=0.5)


@pytest.mark.parametrize("slab", [2, 4, 8])
@pytest.mark.parametrize("pixels", [(0.05, 0.0499), (0.05, 0.0501), (0.08, 0.06)])
def test_rows_and_residency(slab, pixels):
    import paper_2101_05031_gb300 as cs
    jobs, want = [], []
    for k, px in enumerate(pixels):
        lat = _lattice(cs, k)
        d = dict(z0=0.13, dz=0.27, n_layers=11 - k, x0=-0.3, y0=-0.2, nx=int(6.6 / px) + k,
                 ny=int(5.5 / px), pixel=px, edge_ids=True)
        sig = torch.empty((d["n_layers"], d["ny"], d["nx"]), device="cuda")
        c = lat.slice(**d, sigma_out=sig, slab=slab, field_kernel="block")
        jobs.append((lat, d))
        want.append((sig, c))
    rows = 2 if all(0.5 >= 10.0 * px for px in pixels) else 1
    for ctas in range(1, 7):
        b = cs.Batch(jobs, slab=slab, ctas_per_sm=ctas)
        b.run()
        # two rows: CTAs of half the threads, 8 per SM at most
        assert b.info().ctas_per_sm == (min(ctas, 4) if rows == 2 else ctas)
        for j, (sig, c) in enumerate(want):
            assert torch.equal(b.sigma(j), sig)
            got = b.contours(j)
            assert np.array_equal(got.loop_vert_off, c.loop_vert_off)
            assert np.array_equal(got.xy, c.xy) and np.array_equal(got.edge_id, c.edge_id)
        b.close()


def test_tuned_candidates_are_different_residencies():
    import paper_2101_05031_gb300 as cs
    lat = _lattice(cs, 5)
    d = dict(z0=0.13, dz=0.27, n_layers=11, x0=-0.3, y0=-0.2, nx=140, ny=110, pixel=0.045)
    info = cs.Batch([(lat, d)], autotune=True).info()
    tried = [tuple(int(getattr(info, "cand_" + k)[i]) for k in ("kernel", "tile", "slab", "ctas", "stage"))
             for i in range(info.n_candidates)]
    assert len(set(tried)) == len(tried)
    assert all(c <= 4 for _, _, _, c, _ in tried)
    assert (info.field_kernel, info.tile, info.slab, info.ctas_per_sm, info.stage_records) in tried
