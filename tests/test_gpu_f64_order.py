"""FP64 steps at a loose tolerance keep their order of additions.

A CG run that stops at 1e-7 magnifies the rounding of its sums: with the sums in another order (or
r.z taken in parts, or the averaged off-diagonals of K^mech's blocks) the displacement of two steps moves
by 1e-9 to 2e-8 of itself.  So an FP64 context above the tolerance of the fast forms (1e-10) keeps one
arithmetic, and its results are compared with recorded ones: the displacement at eight nodes after two
steps, from the separate kernels with one tree per value, nine values per block and z stored.

Tolerance: the same operations in the same order give the same bits; 1e-12 of the largest value is below
what a rounding difference comes out as.
"""
import numpy as np
import pytest

from paper_2510_09812_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

RECORDED = {
    ((16, 16, 4), 3): [
        (-3.898475034640397e-05, 9.775452867064684e-07, -1.9669361245074054e-05),
        (2.174306919843161e-06, 2.064553808897854e-05, -6.540843834424939e-06),
        (-4.138690041101829e-05, 1.67177975558373e-05, -2.037912437313484e-05),
        (-7.863091647222271e-07, 3.1689643911056475e-05, -1.1359839783252096e-05),
        (-2.7977054734169193e-05, 4.3229450952533984e-05, -2.925685559658142e-05),
        (-1.6711979954130124e-05, 1.536734783704405e-05, -7.708540088977076e-06),
        (-3.330378816332459e-05, 1.5936817087330238e-05, -2.5733415433000313e-05),
        (-8.836514849075287e-06, 1.899380918311061e-05, -8.9371901323819e-06),
    ],
    ((45, 39, 11), 4): [
        (-1.0672355477568073e-05, 1.7094701213818645e-05, 1.5073430977306094e-05),
        (-5.824880330101885e-06, 2.615406149067184e-06, 5.882206745773242e-06),
        (-2.4929994664362053e-05, 3.136251664844679e-05, 9.4529905085065e-06),
        (-1.8849822275267548e-05, -1.462409191242011e-05, -6.905236015254952e-06),
        (-3.211604346930421e-05, 9.094108749853232e-06, -1.730301540719519e-05),
        (1.096793895560332e-05, 1.9762285326829924e-05, 4.3973343470915e-05),
        (-1.769173090547691e-05, 2.4215599234539794e-06, -1.6739514100591027e-05),
        (-2.2438569705827335e-05, 2.182390209898797e-06, 1.4275320275474107e-05),
    ],
}


def _ctx(g, cells, prec, rtol, **kw):
    box = tuple(4.0 * c for c in cells)
    mesh = synth.kuhn_box(cells, box, jitter=0.2, seed=5,
                          defects=[dict(kind="sphere", center=tuple(b / 2 for b in box),
                                        radius=0.3 * min(box))])
    return g.Context(mesh, synth.fe_like_material(), 1e-12, 0.5, precision=prec, rtol_gs=rtol,
                     rtol_ms=rtol, rtol_mech=rtol, autotune=False, **kw)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("cells,seed", list(RECORDED))
def test_recorded_displacement(gspm_lib, cells, seed, graph):
    g = gspm_lib
    ctx = _ctx(g, cells, "f64", 1e-7, graph=graph)
    ctx.set_field(g.FIELD_M, synth.random_unit_m(ctx.n, seed))
    assert ctx.step(2, [2e4, -1e4, 5e3])["noconv"] == 0
    u = ctx.get_field(g.FIELD_DISP)
    stride = ctx.n // 8
    want = np.array(RECORDED[cells, seed])
    assert np.abs(u[stride // 2::stride][:8] - want).max() <= 1e-12 * np.abs(u).max()


def test_tolerance_decides_per_call(gspm_lib):
    """One context: fused loops at 1e-10, the separate kernels above it, and back, by set_rtol and by
    the tolerance of an elastic solve; the two agree within the looser tolerance."""
    g = gspm_lib
    cells, seed = (16, 16, 4), 3
    ctx = _ctx(g, cells, "f64", 1e-10)
    m = synth.random_unit_m(ctx.n, seed)
    z = np.zeros((ctx.n, 3))
    out, launches = [], []
    for rtol in (1e-10, 1e-7, 1e-10):
        ctx.set_rtol(rtol, rtol, rtol)
        for f, v in ((g.FIELD_M, m), (g.FIELD_U, z[:, 0].copy()), (g.FIELD_DISP, z),
                     (g.FIELD_DISP_PREV, z)):
            ctx.set_field(f, v)
        n0 = ctx.launch_count()
        assert ctx.step(2, [2e4, -1e4, 5e3])["noconv"] == 0
        launches.append(ctx.launch_count() - n0)
        out.append(ctx.get_field(g.FIELD_DISP))
    assert launches[0] == launches[2] and launches[1] > 4 * launches[0]
    assert np.array_equal(out[0], out[2])
    top = np.abs(out[0]).max()
    assert 0 < np.abs(out[0] - out[1]).max() < 1e-5 * top
    stride = ctx.n // 8
    assert np.abs(out[1][stride // 2::stride][:8] - RECORDED[cells, seed]).max() <= 1e-12 * top
    loose, tight = (ctx.solve_elastic(m, x0_mode=0, rtol=r)[0].copy() for r in (1e-7, 1e-10))
    n0 = ctx.launch_count()
    ctx.solve_elastic(m, x0_mode=0, rtol=1e-10)
    n1 = ctx.launch_count()
    ctx.solve_elastic(m, x0_mode=0, rtol=1e-7)
    assert ctx.launch_count() - n1 > 4 * (n1 - n0)
    assert np.abs(loose - tight).max() < 1e-5 * np.abs(tight).max()
