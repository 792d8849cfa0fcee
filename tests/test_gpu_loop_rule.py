"""Steps whose scalar solves run fused while K^mech is solved by the separate kernels.

That is so where K^mech has no symmetric blocks (faces that do not match to rounding: nine values per
block) and where an iteration of it streams more than the L2 holds (by size, or by a fine coarse space).
References: ordering "none" (no fused loops at all).  FP64 solves to 1e-12 agree within the CG error
(1e-9 of a field's largest value), mixed steps at 1e-7 within the mixed-precision bound of 1e-4 rad;
graph and direct launches run the same kernels: equal bits, equal iteration counts.
"""
import numpy as np
import pytest

from paper_2510_09812_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _mesh(cells, make=synth.kuhn_box, mismatch=0.0):
    box = tuple(4.0 * c for c in cells)
    mesh = make(cells, box, jitter=0.0 if mismatch else 0.2, seed=5,
                defects=[dict(kind="sphere", center=tuple(b / 2 for b in box),
                              radius=0.3 * min(box))])
    if mismatch:
        top = mesh.coords[:, 2] == mesh.box_hi[2]
        inner = top & (mesh.coords[:, 1] > 0) & (mesh.coords[:, 1] < box[1])
        mesh.coords[inner, 1] += mismatch * np.random.default_rng(4).choice((-1.0, 1.0), inner.sum())
    return mesh


def _ctx(g, mesh, prec, rtol, **kw):
    return g.Context(mesh, synth.fe_like_material(), 1e-12, 0.5, precision=prec, rtol_gs=rtol,
                     rtol_ms=rtol, rtol_mech=rtol, autotune=False, **kw)


def _unit(m):
    mag = np.linalg.norm(m, axis=1) > 0.5
    return m[mag] / np.linalg.norm(m[mag], axis=1, keepdims=True)


def _compare(g, mesh, prec, **kw):
    rtol = 1e-12 if prec == "f64" else 1e-7
    m0 = synth.random_unit_m(mesh.n_unique, 6)
    z = np.zeros((mesh.n_unique, 3))
    runs = []
    ctx = _ctx(g, mesh, prec, rtol, **kw)
    none = {k: v for k, v in kw.items() if k != "coarse_nodes"}
    for c, graph in ((ctx, False), (ctx, True), (_ctx(g, mesh, prec, rtol, ordering="none", **none), False)):
        c.set_graph(graph)
        c.set_true_residual(True)
        for f, v in ((g.FIELD_M, m0), (g.FIELD_U, z[:, 0].copy()), (g.FIELD_DISP, z),
                     (g.FIELD_DISP_PREV, z)):
            c.set_field(f, v)
        n0 = c.launch_count()
        st = c.step(2, [2e4, -1e4, 5e3])
        n1 = c.launch_count()
        assert st["noconv"] == 0
        # (drifts from the recursive residual by rounding; a wrong operator is off by far more)
        assert 0.0 <= st["true_res_mech_last"] < 100 * rtol
        fields = [c.get_field(f) for f in (g.FIELD_M, g.FIELD_U)]
        runs.append((st, n1 - n0, fields + [c.solve_elastic(m0, x0_mode=0, rtol=rtol)[0].copy()]))
    (sd, nd, fd), (sg, ng, fg), (sn, nn, fn) = runs
    # kernels per iteration for K^mech, not for K^ms (whose iterations the reference has in kernels)
    assert nd > 3 * sd["it_mech"]
    if "coarse_nodes" not in kw:
        assert nd < nn - sn["it_ms"]
    for key in ("it_ms", "it_mech", "it_gs", "it_ms_last", "it_mech_last"):
        assert sd[key] == sg[key]
    for x, y in zip(fd, fg):
        assert np.array_equal(x, y)
    if prec == "f64":
        for x, y in zip(fd, fn):
            assert np.abs(x - y).max() <= 1e-9 * np.abs(y).max()
    else:
        assert np.linalg.norm(_unit(fd[0]) - _unit(fn[0]), axis=1).max() < 1e-4


@pytest.mark.parametrize("prec", ["f64", "mixed"])
@pytest.mark.parametrize("make", [synth.kuhn_box, synth.hex_box])
def test_faces_that_do_not_match(gspm_lib, prec, make):
    _compare(gspm_lib, _mesh((13, 11, 9), make, mismatch=4e-4), prec, wrap_tol=2e-3)


@pytest.mark.parametrize("prec", ["f64", "mixed"])
def test_fine_coarse_space(gspm_lib, prec):
    """40,000 nodes in 2,500 aggregates: the inverse of the coarse operator alone is 450 MB in FP64 and
    112 MB in bfloat16."""
    _compare(gspm_lib, _mesh((50, 40, 20)), prec, coarse_nodes=16)


def test_large_mesh(gspm_lib):
    _compare(gspm_lib, _mesh((96, 96, 40)), "mixed")
