"""Two-level CG in separate kernels with z never stored (aggregates that are runs of rows).

It runs where the fused loops do not: above 400,000 nodes (mixed precision), and in batches of more meshes than the GPU
has SMs.  References: the same systems with ordering "none" (aggregates that are not runs of rows,
z stored) and each mesh of a batch alone.  FP64 solves to 1e-12 agree within the CG error (1e-9 of
a field's largest value), mixed steps at 1e-7 within the mixed-precision bound of 1e-4 rad; replayed
graphs and direct launches run the same kernels, so they agree bit for bit.

Sizes: meshes of less than a slice, of a few rows past a slice or a four-row pack, of one aggregate
and of many; work items that start within an aggregate and aggregates that lie within one warp's rows.
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


def _ctx(g, mesh, prec, rtol, **kw):
    return g.Context(mesh, synth.fe_like_material(), 1e-12, 0.5, precision=prec, rtol_gs=rtol,
                     rtol_ms=rtol, rtol_mech=rtol, autotune=False, **kw)


def _unit(m):
    mag = np.linalg.norm(m, axis=1) > 0.5
    return m[mag] / np.linalg.norm(m[mag], axis=1, keepdims=True)


@pytest.mark.parametrize("prec,rtol", [("f64", 1e-12), ("mixed", 1e-7)])
@pytest.mark.parametrize("coarse", [0, 24])
def test_many_small_meshes(gspm_lib, prec, rtol, coarse):
    g = gspm_lib
    sizes = [(3, 3, 3), (4, 4, 2), (5, 4, 5), (7, 5, 3), (9, 8, 7), (16, 15, 11)]
    meshes = [_mesh(sizes[k % len(sizes)], k % 12) for k in range(170)]
    fields = np.array([[1e4 * (k % 3), -5e3 * (k % 2), 2e4] for k in range(len(meshes))])
    m0 = [synth.random_unit_m(m.n_unique, 40 + k % 12) for k, m in enumerate(meshes)]
    kw = dict(coarse_nodes=coarse) if coarse else {}
    out = []
    for graph in (False, True):
        ctx = _ctx(g, meshes, prec, rtol, graph=graph, **kw)
        ctx.set_field(g.FIELD_M, np.concatenate(m0))
        assert all(st["noconv"] == 0 for st in ctx.batch_step(2, fields))
        out.append([ctx.get_field(f) for f in (g.FIELD_M, g.FIELD_U, g.FIELD_DISP, g.FIELD_STRAIN)])
        offs = [ctx.segment(k) for k in range(len(meshes))]
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    for k in list(range(6)) + [169]:
        one = _ctx(g, meshes[k], prec, rtol)
        one.set_field(g.FIELD_M, m0[k])
        one.step(2, fields[k])
        off, cnt = offs[k]
        if prec == "f64":
            for f, got in zip((g.FIELD_M, g.FIELD_U, g.FIELD_DISP, g.FIELD_STRAIN), out[0]):
                want = one.get_field(f)
                assert np.abs(got[off:off + cnt] - want).max() <= 1e-9 * max(np.abs(want).max(), 1e-300)
        else:
            a, b = (_unit(x) for x in (out[0][0][off:off + cnt], one.get_field(g.FIELD_M)))
            assert np.linalg.norm(a - b, axis=1).max() < 1e-4


def test_one_large_mesh(gspm_lib):
    """608,256 nodes: items start within aggregates of about 150 rows."""
    g = gspm_lib
    mesh = _mesh((96, 96, 66), 3)
    m0 = synth.random_unit_m(mesh.n_unique, 8)
    out = []
    for kw in (dict(), dict(graph=True), dict(ordering="none")):
        ctx = _ctx(g, mesh, "mixed", 1e-7, **kw)
        ctx.set_field(g.FIELD_M, m0)
        assert ctx.step(2, [2e4, 0.0, 0.0])["noconv"] == 0
        out.append(ctx.get_field(g.FIELD_M))
        ctx.close()
    assert np.array_equal(out[0], out[1])
    a, b = (_unit(o) for o in (out[0], out[2]))
    assert np.linalg.norm(a - b, axis=1).max() < 1e-4
