"""Fused FP64 loops at the limit of shared memory, with the rest of the state in global memory.

A block's dynamic shared memory and the kernel's static part (4,640 bytes in the FP64 two-level loops)
share 232,448 bytes.  The meshes are ones whose vectors would ask for 227,824 and 228,304 bytes.
Reference: the separate kernels (ordering "none").  Both stop at 1e-10, so they agree within that times
the condition number of these systems (below 1e4): 1e-6 of the largest value.
"""
import numpy as np
import pytest

from paper_2510_09812_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cells", [(78, 46, 68), (94, 66, 40)])
def test_f64_step_and_elastic_solve(gspm_lib, cells):
    g = gspm_lib
    box = tuple(4.0 * c for c in cells)
    mesh = synth.kuhn_box(cells, box, jitter=0.2, seed=5,
                          defects=[dict(kind="sphere", center=tuple(b / 2 for b in box),
                                        radius=0.3 * min(box))])
    m0 = synth.random_unit_m(mesh.n_unique, 6)
    out, launches = [], []
    for ordering in ("aggregate", "none"):
        ctx = g.Context(mesh, synth.fe_like_material(), 1e-12, 0.5, precision="f64", rtol_gs=1e-10,
                        rtol_ms=1e-10, rtol_mech=1e-10, autotune=False, ordering=ordering)
        ctx.set_field(g.FIELD_M, m0)
        n0 = ctx.launch_count()
        assert ctx.step(1, [2e4, -1e4, 5e3])["noconv"] == 0
        launches.append(ctx.launch_count() - n0)
        u, it, rel, code = ctx.solve_elastic(m0, x0_mode=0)
        assert code == 0 and it > 10
        out.append([ctx.get_field(f) for f in (g.FIELD_M, g.FIELD_U)] + [u.copy()])
        ctx.close()
    assert launches[0] < launches[1] / 4
    for x, y in zip(*out):
        assert np.abs(x - y).max() <= 1e-6 * np.abs(y).max()
