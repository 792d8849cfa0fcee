"""Storage of the K^mech blocks: the upper triangle of a symmetric block (6 values) on every mesh
whose periodic faces match, all nine values otherwise.

A mesh whose matching face nodes differ in their in-plane coordinates by less than wrap_tol has
blocks that are not symmetric (the two sides of the face do not coincide); storing them as
symmetric ones would move the product by about the mismatch over the node spacing (1e-4 here).
Tolerance: the operator parity one (1e-13 FP64, 2e-6 mixed: FP32 rounding of values and operands).
"""
import numpy as np
import pytest

from oracle.gspm import System
from oracle.mesh import WrappedMesh
from paper_2510_09812_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("f64", 1e-13), ("mixed", 2e-6)])
@pytest.mark.parametrize("make", [synth.kuhn_box, synth.hex_box])
@pytest.mark.parametrize("mismatch", [0.0, 4e-4])
def test_block_product_matches_oracle(gspm_lib, prec, tol, make, mismatch):
    g = gspm_lib
    wrap_tol = 2e-3
    mesh = make((7, 5, 4), (28.0, 20.0, 16.0), jitter=0.0)     # 140 rows: a ragged last slice
    top = mesh.coords[:, 2] == mesh.box_hi[2]
    inner = top & (mesh.coords[:, 1] > 0) & (mesh.coords[:, 1] < 20.0)
    sign = np.random.default_rng(4).choice((-1.0, 1.0), inner.sum())
    mesh.coords[inner, 1] += mismatch * sign
    wm = WrappedMesh(mesh.coords, mesh.tets, mesh.elem_magnetic, mesh.box_lo, mesh.box_hi,
                     tol=wrap_tol)
    assert wm.n == 140
    s = System(wm, synth.fe_like_material(), 1e-12, 0.5)
    blocks = s.K_mech_raw.tobsr((3, 3)).data
    asym = np.abs(blocks - blocks.transpose(0, 2, 1)).max() / np.abs(blocks).max()
    assert asym > 1e-7 if mismatch else asym < 1e-15
    ctx = g.Context(mesh, synth.fe_like_material(), 1e-12, 0.5, precision=prec, wrap_tol=wrap_tol,
                    plain_cg=True)
    x = np.random.default_rng(5).standard_normal((wm.n, 3))
    want = (s.K_mech @ x.ravel()).reshape(-1, 3)
    got = ctx.apply(g.OP_K_MECH, x)
    assert np.abs(got - want).max() < tol * np.abs(want).max()
