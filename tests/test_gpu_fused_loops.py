"""CG loops fused into one cooperative kernel (default up to a size) against the separate kernels.

The separate kernels run where the fused loops do not apply: with the two-level preconditioner, for
instance, when the aggregates are not runs of rows (ordering "none" and
several aggregates).  Both are CG on the same systems
with the same stopping test, so FP64 solves to 1e-12 agree within the CG error (1e-9 of a field's
largest value: 1e-12 times the condition of these small systems, with room), and mixed steps at 1e-7
within the mixed-precision bound of 1e-4 rad.

Sizes: one slice of 32 rows and a ragged one; every block one slice shared by sixteen warps; one row
slice more than the 152 blocks (blocks of one and of two slices); around sixteen slices per block,
where warps stop sharing slices; state partly outside shared memory; meshes of a batch of very
different sizes, so that groups of blocks stop at different times.
"""
import numpy as np
import pytest

from paper_2510_09812_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _mesh(cells, seed=5, make=synth.kuhn_box):
    box = tuple(4.0 * c for c in cells)
    return make(cells, box, jitter=0.2, seed=seed,
                defects=[dict(kind="sphere", center=tuple(b / 2 for b in box),
                              radius=0.3 * min(box))])


def _ctx(g, mesh, prec, rtol, **kw):
    return g.Context(mesh, synth.fe_like_material(), 1e-12, 0.5, precision=prec, rtol_gs=rtol,
                     rtol_ms=rtol, rtol_mech=rtol, autotune=False, **kw)


def _fields(g, ctx):
    return [ctx.get_field(f) for f in (g.FIELD_M, g.FIELD_U, g.FIELD_DISP, g.FIELD_STRAIN)]


def _close(a, b, tol):
    for x, y in zip(a, b):
        assert np.abs(x - y).max() <= tol * max(np.abs(y).max(), 1e-300)


@pytest.mark.parametrize("make", [synth.kuhn_box, synth.hex_box])
@pytest.mark.parametrize("cells,coarse", [((4, 4, 2), 8), ((5, 4, 5), 16), ((8, 8, 8), 64),
                                          ((21, 19, 13), 64), ((20, 19, 13), 0), ((41, 40, 25), 0)])
def test_fused_loops_match_separate_kernels(gspm_lib, cells, coarse, make):
    g = gspm_lib
    mesh = _mesh(cells, make=make)
    m0 = synth.random_unit_m(mesh.n_unique, 6)
    out, launches = [], []
    for ordering in ("aggregate", "none"):
        ctx = _ctx(g, mesh, "f64", 1e-12, ordering=ordering, coarse_nodes=coarse)
        ctx.set_field(g.FIELD_M, m0)
        n0 = ctx.launch_count()
        st = ctx.step(2, [2e4, -1e4, 5e3])
        launches.append(ctx.launch_count() - n0)
        assert st["noconv"] == 0
        out.append(_fields(g, ctx))
    assert launches[0] < launches[1] / 4          # a few launches per solve, not per iteration
    _close(out[0], out[1], 1e-9)


@pytest.mark.parametrize("kw", [dict(plain_cg=True), dict(pinned_cg=True)])
@pytest.mark.parametrize("cells", [(5, 4, 5), (21, 19, 13), (41, 40, 25)])
def test_fused_plain_forms_match_preconditioned(gspm_lib, cells, kw):
    g = gspm_lib
    mesh = _mesh(cells)
    m0 = synth.random_unit_m(mesh.n_unique, 7)
    out = []
    for k in (kw, dict(ordering="none", coarse_nodes=16 if cells[0] < 8 else 0)):
        ctx = _ctx(g, mesh, "f64", 1e-12, **k)
        ctx.set_field(g.FIELD_M, m0)
        assert ctx.step(1, [0.0, 2e4, 0.0])["noconv"] == 0
        out.append(_fields(g, ctx))
    _close(out[0], out[1], 1e-9)


@pytest.mark.parametrize("cells", [(8, 8, 8), (41, 40, 25), (96, 96, 40)])
def test_fused_mixed_steps_within_angle(gspm_lib, cells):
    """Up to 368,640 nodes, where a block's vectors no longer fit its shared memory."""
    g = gspm_lib
    mesh = _mesh(cells)
    m0 = synth.random_unit_m(mesh.n_unique, 8)
    out = []
    for ordering in ("aggregate", "none"):
        ctx = _ctx(g, mesh, "mixed", 1e-7, ordering=ordering, coarse_nodes=64 if cells[0] < 9 else 0)
        ctx.set_field(g.FIELD_M, m0)
        assert ctx.step(2, [2e4, 0.0, 0.0])["noconv"] == 0
        out.append(ctx.get_field(g.FIELD_M))
        ctx.close()
    mag = np.linalg.norm(out[0], axis=1) > 0.5
    a, b = (o[mag] / np.linalg.norm(o[mag], axis=1, keepdims=True) for o in out)
    assert np.linalg.norm(a - b, axis=1).max() < 1e-4      # the chord, for unit vectors the angle


@pytest.mark.parametrize("prec,tol", [("f64", 1e-9), ("mixed", 1e-4)])
def test_fused_batch_matches_each_mesh_alone(gspm_lib, prec, tol):
    g = gspm_lib
    meshes = [_mesh((4, 4, 2), 1), _mesh((30, 28, 11), 2), _mesh((7, 5, 3), 3), _mesh((12, 12, 9), 4)]
    fields = np.array([[1e4, 0, 0], [0, 2e4, 0], [0, 0, -1e4], [5e3, 5e3, 0]])
    rtol = 1e-12 if prec == "f64" else 1e-7
    ms = [synth.random_unit_m(m.n_unique, 20 + k) for k, m in enumerate(meshes)]
    batch = _ctx(g, meshes, prec, rtol)
    batch.set_field(g.FIELD_M, np.concatenate(ms))
    for st in batch.batch_step(2, fields):
        assert st["noconv"] == 0
    got = _fields(g, batch)
    for k, mesh in enumerate(meshes):
        one = _ctx(g, mesh, prec, rtol, ordering="none", coarse_nodes=max(8, mesh.n_unique // 16))
        one.set_field(g.FIELD_M, ms[k])
        one.step(2, fields[k])
        off, cnt = batch.segment(k)
        _close([f[off:off + cnt] for f in got], _fields(g, one), tol)


def test_zero_right_hand_side_and_reuse(gspm_lib):
    """A uniform m in a mesh without defects has b = 0 up to rounding (nothing to solve); a solve
    before and after it on the same context gives the same result."""
    g = gspm_lib
    mesh = synth.kuhn_box((12, 10, 6), (48.0, 40.0, 24.0), jitter=0.0)
    n = mesh.n_unique
    ctx = _ctx(g, mesh, "f64", 1e-12)
    m = synth.random_unit_m(n, 9)
    first = ctx.solve_elastic(m, x0_mode=0)[0].copy()
    zero = np.zeros((n, 3))
    u, it, rel, code = ctx.solve_elastic(zero, x0_mode=0)     # E0 uniform, b exactly 0 or rounding
    assert np.abs(u).max() < 1e-6 * np.abs(first).max() or it == 0
    again = ctx.solve_elastic(m, x0_mode=0)[0]
    assert np.array_equal(first, again)
