"""Fused CG loops on batches whose meshes do not keep step.

Meshes of a batch number their exchanges themselves: one that starts converged, or needs fewer
iterations, runs out of step with the others, solve by solve.  A converged start is made by solving to
1e-13 and then asking for 1e-12 from that solution.  Each mesh is compared with a context of its own
(FP64 to 1e-12: within the CG error, 1e-9 of the largest value; the separate kernels, ordering "none").
"""
import numpy as np
import pytest

from paper_2510_09812_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _mesh(cells, seed):
    box = tuple(4.0 * c for c in cells)
    return synth.kuhn_box(cells, box, jitter=0.2, seed=seed,
                          defects=[dict(kind="sphere", center=tuple(b / 2 for b in box),
                                        radius=0.3 * min(box))])


def _ctx(g, mesh, rtol=1e-12, material=None, **kw):
    return g.Context(mesh, material or synth.fe_like_material(), 1e-12, 0.5, precision="f64",
                     rtol_gs=rtol, rtol_ms=rtol, rtol_mech=rtol, autotune=False, **kw)


def _close(a, b, tol=1e-9):
    assert np.abs(a - b).max() <= tol * max(np.abs(b).max(), 1e-300)


def test_meshes_that_start_converged(gspm_lib):
    """All meshes but one start converged, in turn, between steps that move every mesh on by a
    different number of exchanges."""
    g = gspm_lib
    cells = [(16, 16, 8), (16, 16, 8), (9, 8, 7), (30, 28, 11)]
    meshes = [_mesh(c, k) for k, c in enumerate(cells)]
    ms = [synth.random_unit_m(m.n_unique, 20 + k) for k, m in enumerate(meshes)]
    batch = _ctx(g, meshes)
    off = [batch.segment(k) for k in range(len(meshes))]
    alone = [_ctx(g, m, ordering="none", coarse_nodes=max(8, m.n_unique // 16)) for m in meshes]
    fields = np.array([[1e4, 0, 0], [0, 2e4, 0], [0, 0, -1e4], [5e3, 5e3, 0]])
    cur = np.concatenate(ms)
    batch.set_field(g.FIELD_M, cur)
    for k, a in enumerate(alone):
        a.set_field(g.FIELD_M, ms[k])
    for rnd in range(len(meshes)):
        first = batch.solve_elastic(cur, x0_mode=0, rtol=1e-13)[0].copy()
        o, n = off[rnd]
        m2 = cur.copy()
        m2[o:o + n] = synth.random_unit_m(n, 50 + rnd)
        u, it, rel, code = batch.solve_elastic(m2, x0_mode=1, rtol=1e-12)
        assert it > 0 and code == 0
        same = np.ones(len(u), bool)
        same[o:o + n] = False
        # nothing to do there but taking off the mean and the pinned value again: a few roundings
        assert np.abs(u[same] - first[same]).max() <= 8 * 2.0 ** -53 * np.abs(first).max()
        _close(u[o:o + n], alone[rnd].solve_elastic(m2[o:o + n], x0_mode=0, rtol=1e-12)[0])
        cur = m2
        assert all(st["noconv"] == 0 for st in batch.batch_step(1, fields))
        got = [batch.get_field(f) for f in (g.FIELD_M, g.FIELD_U, g.FIELD_DISP)]
        for k, a in enumerate(alone):
            assert a.step(1, fields[k])["noconv"] == 0
            for x, f in zip(got, (g.FIELD_M, g.FIELD_U, g.FIELD_DISP)):
                _close(x[off[k][0]:off[k][0] + off[k][1]], a.get_field(f))


@pytest.mark.parametrize("count", [1, 3])
def test_zero_right_hand_side_writes_zero(gspm_lib, count):
    """No magnetostriction: b = 0 exactly, so the solution is 0 whatever the start was."""
    g = gspm_lib
    mat = dict(synth.fe_like_material(), lambda100=0.0, lambda111=0.0)
    meshes = [_mesh((12, 10, 6 + k), k) for k in range(count)]
    ctx = _ctx(g, meshes if count > 1 else meshes[0], material=mat)
    n = ctx.n
    ctx.set_field(g.FIELD_DISP, np.random.default_rng(3).standard_normal((n, 3)))
    u, it, rel, code = ctx.solve_elastic(synth.random_unit_m(n, 9), x0_mode=1)
    assert it == 0 and code == 0
    assert not u.any()
