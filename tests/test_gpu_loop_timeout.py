"""A wait of a fused CG loop that runs out (a limit of one poll, which no exchange meets).

The call returns GSPM_ETIMEOUT although many steps were queued, and the same context then solves
with the separate kernels: FP64 to 1e-12 like a fresh context within the CG error (1e-9 of a field's
largest value).
"""
import time

import numpy as np
import pytest

from paper_2510_09812_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _mesh(cells, seed=5):
    box = tuple(4.0 * c for c in cells)
    return synth.kuhn_box(cells, box, jitter=0.2, seed=seed,
                          defects=[dict(kind="sphere", center=tuple(b / 2 for b in box),
                                        radius=0.3 * min(box))])


def _ctx(g, mesh, graph):
    return g.Context(mesh, synth.fe_like_material(), 1e-12, 0.5, precision="f64", rtol_gs=1e-12,
                     rtol_ms=1e-12, rtol_mech=1e-12, autotune=False, graph=graph)


def _start(g, ctx, m):
    z = np.zeros((ctx.n, 3))
    for f, v in ((g.FIELD_M, m), (g.FIELD_U, z[:, 0].copy()), (g.FIELD_DISP, z),
                 (g.FIELD_DISP_PREV, z)):
        ctx.set_field(f, v)


def _fails(g, call):
    t = time.monotonic()
    with pytest.raises(g.GSPMError) as e:
        call()
    assert e.value.code == g.ETIMEOUT
    return time.monotonic() - t


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("batch", [False, True])
def test_step_fails_then_goes_on(gspm_lib, batch, graph):
    g = gspm_lib
    meshes = [_mesh((21, 19, 13)), _mesh((8, 8, 8), 6)][:2 if batch else 1]
    mesh = meshes if batch else meshes[0]
    H = [2e4, -1e4, 5e3]
    ctx, ref = _ctx(g, mesh, graph), _ctx(g, mesh, graph)
    m = synth.random_unit_m(ctx.n, 6)
    step = (lambda c, k: c.batch_step(k, np.array([H, H]))) if batch else (lambda c, k: c.step(k, H))
    launches = []
    for c in (ref, ctx):
        _start(g, c, m)
        n0 = c.launch_count()
        step(c, 2)
        launches.append(c.launch_count() - n0)
    assert launches[0] == launches[1]
    ctx.set_wait_limit(1)
    assert _fails(g, lambda: step(ctx, 300)) < 20.0
    _start(g, ctx, m)
    n0 = ctx.launch_count()
    step(ctx, 2)
    assert ctx.launch_count() - n0 > 4 * launches[0]        # kernels per iteration, not per solve
    for f in (g.FIELD_M, g.FIELD_U, g.FIELD_DISP):
        a, b = ctx.get_field(f), ref.get_field(f)
        assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()


def test_elastic_solve_fails_then_goes_on(gspm_lib):
    g = gspm_lib
    mesh = _mesh((21, 19, 13))
    ctx = _ctx(g, mesh, False)
    m = synth.random_unit_m(ctx.n, 6)
    want = ctx.solve_elastic(m, x0_mode=0)[0].copy()
    ctx.set_wait_limit(1)
    _fails(g, lambda: ctx.solve_elastic(m, x0_mode=0))
    u, it, rel, code = ctx.solve_elastic(m, x0_mode=0)
    assert code == 0 and it > 10
    assert np.abs(u - want).max() <= 1e-9 * np.abs(want).max()


def test_limit_is_kept_and_restored(gspm_lib):
    """An ample limit changes nothing; 0 restores the default."""
    g = gspm_lib
    mesh = _mesh((8, 8, 8))
    ctx = _ctx(g, mesh, True)
    m = synth.random_unit_m(ctx.n, 6)
    out = []
    for polls in (1 << 20, 0):
        ctx.set_wait_limit(polls)
        _start(g, ctx, m)
        assert ctx.step(2, [2e4, 0.0, 0.0])["noconv"] == 0
        out.append(ctx.get_field(g.FIELD_DISP))
    assert np.array_equal(*out)
