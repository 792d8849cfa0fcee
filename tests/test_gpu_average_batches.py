"""Volume averages of batches: more meshes than a grid has rows, and meshes of very uneven size.

Sums of at most 131,072 FP64 products with weights that add up to one: 1e-13 of the largest value.
"""
import numpy as np
import pytest

from paper_2510_09812_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _ctx(g, meshes):
    return g.Context(meshes, synth.fe_like_material(), 1e-12, 0.5, precision="f64", plain_cg=True,
                     autotune=False)


def test_more_meshes_than_grid_rows(gspm_lib):
    g = gspm_lib
    count = 65600
    ctx = _ctx(g, [synth.kuhn_box((2, 2, 2), (8.0, 8.0, 8.0))] * count)   # 8 nodes, equal weights
    assert ctx.n == 8 * count
    f = np.random.default_rng(1).standard_normal((ctx.n, 3))
    got = ctx.volume_avg(f)
    want = f.reshape(count, 8, 3).mean(1)
    assert np.abs(np.asarray(got).reshape(count, 3) - want).max() <= 1e-13 * np.abs(f).max()
    # 2.1M rows (each mesh a slice of its own) of 8 entries with some 35 values, 0.6 KB of scratch a row:
    # 6 GB at most; partials of 78 KB for each mesh would be 5 GB more
    assert ctx.info()["device_bytes"] < 6 << 30
    ctx.close()


@pytest.mark.parametrize("nc", [1, 2, 6, 9])
def test_uneven_meshes(gspm_lib, nc):
    """One block, a few, and the most that a mesh gets; the same as each mesh alone."""
    g = gspm_lib
    cells = [(4, 3, 2), (64, 64, 32), (13, 11, 9), (40, 20, 10)]
    meshes = [synth.kuhn_box(c, tuple(4.0 * x for x in c), jitter=0.2, seed=k)
              for k, c in enumerate(cells)]
    ctx = _ctx(g, meshes)
    f = np.random.default_rng(2).standard_normal((ctx.n, nc))
    for _ in range(2):                                   # the counters are left at zero
        got = np.asarray(ctx.volume_avg(f)).reshape(len(cells), nc)
        for k, mesh in enumerate(meshes):
            o, n = ctx.segment(k)
            one = _ctx(g, mesh)
            want = np.asarray(one.volume_avg(f[o:o + n])).reshape(nc)
            one.close()
            assert np.abs(got[k] - want).max() <= 1e-13 * np.abs(f).max()
    ctx.close()
