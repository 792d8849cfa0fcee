"""What the framework's users run, as measurable cases.

A case names a workload of the public binding (``paper_2510_09812_gb300.gspm``): time steps of one
mesh from a few hundred to three million nodes, batches of uneven meshes, the stand-alone elastic
solve, the learned warm start's training gradient and the volume averages.  Meshes, materials and
weights are the repository's own synthetic ones; magnetisations are seeded smooth textures with
noise.  ``exact`` restates each pass in FP64 torch (own assembly, solves to 1e-12).

Mixed-precision contexts keep FP32 state, so their results are kept as float32 here, as a program
that stores or post-processes them would; FP64 contexts return float64.
"""
from __future__ import annotations

import functools
import math
import os

import numpy as np
import torch

from paper_2510_09812_gb300 import gspm, synth

MU0 = 1.25663706212e-6
GAMMA0 = 2.2127615e5
H_NM = 4.0                 # node spacing of every generated box but the 3M-node one
EXACT_NODES = 80_000       # larger meshes take too long to restate in FP64


def listed():
    return [
        # volume average of a small mesh's magnetisation: the smallest call, read every few steps
        dict(name="average_1k", kind="average", cells="16x16x4", recipe="box", ncomp=3),
        # caller-owned arrays of the 3M-node mesh (strain, six components), nothing allocated
        dict(name="average_noalloc_3M", kind="average_noalloc", n=2963088, ncomp=6),
        # the 1,024-node box, the smallest mesh a step is run on: launches and latency only
        dict(name="step_f64_1k", kind="step", cells="16x16x4", recipe="box", precision="f64",
             form="two_level", graph=False, guess="prev", steps=4, dt=1e-12, alpha=0.5,
             rtol=1e-7, field_T=0.0),
        # a mid-size defect mesh with odd, uneven sides in direct launches (host-driven loops)
        dict(name="step_mixed_19k", kind="step", cells="45x39x11", recipe="sphere",
             precision="mixed", form="two_level", graph=False, guess="prev", steps=3, dt=5e-12,
             alpha=0.5, rtol=1e-7, field_T=0.05),
        # the relaxation study: hexahedra, FP64, tight tolerance, replayed graph
        dict(name="step_f64_hex_65k", kind="step", cells="64x64x16", recipe="hex",
             precision="f64", form="two_level", graph=True, guess="extrapolate", steps=2,
             dt=1e-12, alpha=0.15, rtol=1e-10, field_T=2.5e-4),
        # the same in the published form: pinned systems, plain CG
        dict(name="step_f64_pinned_65k", kind="step", cells="64x64x16", recipe="hex",
             precision="f64", form="pinned", graph=False, guess="prev", steps=1, dt=1e-12,
             alpha=0.15, rtol=1e-10, field_T=2.5e-4),
        # the sphere-inclusion workload at its reduced size
        dict(name="step_mixed_65k", kind="step", cells="64x64x16", recipe="sphere",
             precision="mixed", form="two_level", graph=True, guess="prev", steps=3, dt=5e-12,
             alpha=0.5, rtol=1e-7, field_T=2.5e-4),
        # and at its full one (half a million nodes)
        dict(name="step_mixed_524k", kind="step", cells="128x128x32", recipe="sphere",
             precision="mixed", form="two_level", graph=True, guess="extrapolate", steps=2,
             dt=5e-12, alpha=0.5, rtol=1e-7, field_T=2.5e-4),
        # the headline: three million nodes, voids and cuboids, learned guess, reversing field
        dict(name="step_learned_3M", kind="step", cells="228x228x57", recipe="void_cuboids",
             precision="mixed", form="two_level", graph=True, guess="learned", steps=2, dt=5e-12,
             alpha=0.5, rtol=1e-7, field_T=-0.2),
        # sixteen meshes of uneven size under their own fields, advanced together
        dict(name="batch_mixed_16", kind="batch", first=0, count=16, precision="mixed",
             graph=True, steps=1),
        # displacement of one magnetisation from scratch, as the training set is generated
        dict(name="elastic_mixed_150k", kind="elastic", cells="97x83x19", recipe="sphere",
             precision="mixed", rtol=1e-9),
        # loss and gradients of the warm-start network on one stored pair
        dict(name="train_grad_65k", kind="grad", cells="64x64x16", recipe="sphere"),
    ]


def _cells(rng, lo, hi):
    """Uneven cell counts with about lo..hi nodes in all, log-uniform."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ax, ay = rng.uniform(1.0, 4.5), rng.uniform(1.0, 4.5)
    nz = max(4, round((n / (ax * ay)) ** (1.0 / 3.0)))
    ny = max(4, round(ay * nz))
    nx = max(4, round(n / (ny * nz)))
    return "%dx%dx%d" % (nx, ny, nz)


def draw(rng):
    kind = rng.choices(("step", "batch", "elastic", "grad", "average", "average_noalloc"),
                       (9, 2, 3, 2, 1, 1))[0]
    if kind == "average":
        return dict(kind=kind, cells=_cells(rng, 500, 5e5), recipe=rng.choice(("box", "sphere")),
                    ncomp=rng.randint(1, 9))
    if kind == "average_noalloc":
        return dict(kind=kind, n=int(math.exp(rng.uniform(math.log(300), math.log(2.9e6)))),
                    ncomp=rng.randint(1, 9))
    if kind == "batch":
        return dict(kind=kind, first=rng.randint(0, 52), count=rng.randint(2, 11),
                    precision=rng.choice(("mixed", "mixed", "f64")),
                    graph=rng.random() < 0.6, steps=1)
    if kind == "elastic":
        return dict(kind=kind, cells=_cells(rng, 1000, 5e5), recipe="sphere",
                    precision=rng.choice(("mixed", "mixed", "f64")),
                    rtol=rng.choice((1e-7, 1e-9)))
    if kind == "grad":
        return dict(kind=kind, cells=_cells(rng, 1000, 3e5),
                    recipe=rng.choice(("sphere", "hex")))
    precision = rng.choice(("mixed", "mixed", "f64"))
    pinned = rng.random() < 0.15
    cells = _cells(rng, 700, 4e4 if pinned else (1e5 if precision == "f64" else 5e5))
    recipe = rng.choice(("sphere", "sphere", "hex"))
    guess = rng.choice(("prev", "extrapolate", "learned" if precision == "mixed" else "zero"))
    return dict(kind=kind, cells=cells, recipe=recipe, precision=precision,
                form="pinned" if pinned else "two_level", graph=rng.random() < 0.5, guess=guess,
                steps=rng.randint(1, 3), dt=rng.choice((1e-12, 5e-12)),
                alpha=rng.choice((0.15, 0.5)), rtol=1e-10 if precision == "f64" else 1e-7,
                field_T=round(rng.uniform(-0.2, 0.2), 4))


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------

def _sides(case):
    return tuple(int(v) for v in case["cells"].split("x"))


@functools.lru_cache(maxsize=2)
def _mesh(cells, recipe):
    c = tuple(int(v) for v in cells.split("x"))
    box = tuple(H_NM * v for v in c)
    if recipe == "box":
        return synth.kuhn_box(c, box), synth.fe_like_material()
    if recipe == "hex":
        cfg = synth.cuboid_defect_hex_box(n_cells=c, h=H_NM)
    elif recipe == "void_cuboids":
        cfg = synth.void_cuboids_box(n_cells=c)
    else:
        cfg = synth.sphere_inclusion_box(n_cells=c, box=box, radius=0.25 * min(box))
    return cfg["mesh"], cfg["material"]


# A context is what a program keeps for one mesh: loading it costs seconds to half a minute, and
# every state of that mesh is run on it.  The latest two are kept.
@functools.lru_cache(maxsize=2)
def _context(cells, recipe, precision, form, graph, guess, dt, alpha, rtol):
    mesh, material = _mesh(cells, recipe)
    pinned = form == "pinned"
    ctx = gspm.Context(mesh, material, dt, alpha, precision=precision, rtol_gs=rtol,
                       rtol_ms=rtol, rtol_mech=rtol, pinned_cg=pinned, plain_cg=pinned,
                       graph=graph)
    if guess == "learned":
        ctx.mpnn_set_params(_weights())
    ctx.set_x0_mode({"prev": gspm.X0_PREV, "zero": gspm.X0_ZERO,
                     "extrapolate": gspm.X0_EXTRAPOLATE, "learned": gspm.X0_LEARNED}[guess])
    return ctx


@functools.lru_cache(maxsize=1)
def _batch_configs(first, count):
    return [synth.batch_member(i) for i in range(first, first + count)]


@functools.lru_cache(maxsize=1)
def _batch_context(first, count, precision, graph):
    cfgs = _batch_configs(first, count)
    rtol = 1e-10 if precision == "f64" else 1e-7
    return gspm.Context([c["mesh"] for c in cfgs], cfgs[0]["material"], cfgs[0]["dt"],
                        cfgs[0]["alpha"], precision=precision, rtol_gs=rtol, rtol_ms=rtol,
                        rtol_mech=rtol, graph=graph)


def _weights():
    return np.load(os.path.join(os.path.dirname(gspm.__file__), "weights", "warmstart_mpnn.npy"))


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _waves(sides, gen, ncomp, modes=4):
    """[n][ncomp] smooth periodic texture: a few long-wave Fourier modes of random phase."""
    n = [torch.arange(s, dtype=torch.float64, device="cuda") * (2.0 * math.pi / s) for s in sides]
    out = torch.zeros(sides[2], sides[1], sides[0], ncomp, dtype=torch.float64, device="cuda")
    for _ in range(modes):
        k = torch.randint(-2, 3, (3,), generator=gen, device="cuda").double()
        ph = torch.rand(ncomp, generator=gen, device="cuda", dtype=torch.float64) * 2 * math.pi
        am = torch.randn(ncomp, generator=gen, device="cuda", dtype=torch.float64) / modes ** 0.5
        arg = (k[2] * n[2])[:, None, None] + (k[1] * n[1])[None, :, None] + (k[0] * n[0])
        out += am * torch.cos(arg[..., None] + ph)
    return out.reshape(-1, ncomp)


def _magnetisation(sides, gen):
    """Unit vectors: e1 bent by a smooth texture, with a little node-to-node noise."""
    m = 0.6 * _waves(sides, gen, 3)
    m += 0.03 * torch.randn(m.shape, generator=gen, device="cuda", dtype=torch.float64)
    m[:, 0] += 1.0
    return m / m.norm(dim=1, keepdim=True)


def _displacement(sides, gen):
    """A displacement of the size that magnetostriction gives on these boxes (nm)."""
    return 2e-5 * H_NM * 10.0 * _waves(sides, gen, 3)


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "average":
        ctx = _context(case["cells"], case["recipe"], "f64", "pinned", False, "prev", 1e-12, 0.5,
                       1e-7)
        f = 0.5 + torch.randn(ctx.n, case["ncomp"], generator=gen, device="cuda",
                              dtype=torch.float64)
        return dict(kind=kind, ctx=ctx, field=f)
    if kind == "average_noalloc":
        f = 0.5 + torch.randn(case["n"], case["ncomp"], generator=gen, device="cuda",
                              dtype=torch.float64)
        w = 0.5 + torch.rand(case["n"], generator=gen, device="cuda", dtype=torch.float64)
        return dict(kind=kind, field=f, weights=w / w.sum(),
                    out=torch.empty(case["ncomp"], dtype=torch.float64, device="cuda"))
    if kind == "batch":
        cfgs = _batch_configs(case["first"], case["count"])
        ctx = _batch_context(case["first"], case["count"], case["precision"], case["graph"])
        m = torch.cat([_magnetisation(c["mesh"].n_cells, gen) for c in cfgs])
        return dict(kind=kind, ctx=ctx, m=m, steps=case["steps"],
                    fields=np.stack([c["H"] for c in cfgs]), **_buffers(ctx))
    sides = _sides(case)
    if kind == "grad":
        mesh, material = _mesh(case["cells"], case["recipe"])
        ctx = gspm.Context(mesh, material, 5e-12, 0.5, precision="mixed", plain_cg=True,
                           autotune=False)
        ctx.mpnn_set_params(_weights())
        ctx.mpnn_dataset_reserve(1)
        m, u1 = _magnetisation(sides, gen), _displacement(sides, gen)
        u0 = u1 + 0.1 * _displacement(sides, gen)
        ctx.mpnn_dataset_add(m, u1, u0, u1 + 0.1 * _displacement(sides, gen))
        return dict(kind=kind, ctx=ctx)
    m = _magnetisation(sides, gen)
    if kind == "elastic":
        ctx = _context(case["cells"], case["recipe"], case["precision"], "two_level", False,
                       "prev", 5e-12, 0.5, 1e-7)
        return dict(kind=kind, ctx=ctx, m=m, u=torch.empty_like(m), rtol=case["rtol"])
    ctx = _context(case["cells"], case["recipe"], case["precision"], case["form"], case["graph"],
                   case["guess"], case["dt"], case["alpha"], case["rtol"])
    return dict(kind=kind, ctx=ctx, m=m, steps=case["steps"],
                field=[case["field_T"] / MU0, 0.0, 0.0], **_buffers(ctx))


def _buffers(ctx):
    zero = torch.zeros(ctx.n, 3, dtype=torch.float64, device="cuda")
    return dict(zero=zero, zero1=zero[:, 0].contiguous(), m_out=torch.empty_like(zero),
                U_out=torch.empty_like(zero[:, 0]), u_out=torch.empty_like(zero))


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------

def _kept(ctx, t):
    return t.float() if ctx.precision == "mixed" else t


def run(state):
    kind = state["kind"]
    if kind == "average":
        return state["ctx"].volume_avg(state["field"])
    if kind == "average_noalloc":
        return gspm.volume_avg_noalloc(state["field"], state["weights"], state["out"])
    ctx = state["ctx"]
    if kind == "grad":
        loss, grad = ctx.mpnn_loss_grad(0)
        return dict(loss=np.float32(loss), grad=grad)
    if kind == "elastic":
        ctx.solve_elastic(state["m"], state["u"], x0_mode=0, rtol=state["rtol"])
        return _kept(ctx, state["u"])
    # a new state of the mesh: m given, equilibria not known yet; the first step is a cold start
    ctx.set_field(gspm.FIELD_M, state["m"])
    ctx.set_field(gspm.FIELD_U, state["zero1"])
    ctx.set_field(gspm.FIELD_DISP, state["zero"])
    ctx.set_field(gspm.FIELD_DISP_PREV, state["zero"])
    if kind == "batch":
        ctx.batch_step(state["steps"], state["fields"])
    else:
        ctx.step(state["steps"], state["field"])
    ctx.get_field(gspm.FIELD_M, state["m_out"])
    ctx.get_field(gspm.FIELD_U, state["U_out"])
    ctx.get_field(gspm.FIELD_DISP, state["u_out"])
    return dict(m=_kept(ctx, state["m_out"]), U=_kept(ctx, state["U_out"]),
                u=_kept(ctx, state["u_out"]))


# ------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------

def _step_work(n, entries, precision, steps):
    """Per step: every operator (K^mech 9, F and G 3 each, K^ms and three GSPM matrices 1 per
    entry), the columns and the state once; two operations per matrix value.  CG iterations come
    on top, but how many is the solver's business."""
    w = 4 if precision == "mixed" else 8
    values = entries * 19
    return dict(bytes=steps * n * (values * w + 4 * entries + 14 * w),
                flops=steps * n * 2 * values)


def work(case):
    kind = case["kind"]
    if kind == "average_noalloc":
        return dict(bytes=8 * case["n"] * (case["ncomp"] + 1),
                    flops=2 * case["n"] * case["ncomp"])
    if kind == "batch":
        n = sum(16 * max(2, round((_member_nodes(i) / 16.0) ** (1.0 / 3.0))) ** 3
                for i in range(case["first"], case["first"] + case["count"]))
        return _step_work(n, 15, case["precision"], case["steps"])
    sides = _sides(case)
    n = sides[0] * sides[1] * sides[2]
    entries = 27 if case["recipe"] == "hex" else 15
    if kind == "average":
        return dict(bytes=8 * n * (case["ncomp"] + 1), flops=2 * n * case["ncomp"])
    if kind == "elastic":
        w = 4 if case["precision"] == "mixed" else 8
        return dict(bytes=n * (entries * (12 * w + 4) + 6 * 8), flops=n * entries * 24)
    if kind == "grad":
        # forward: three layers of 2 x 128 x 64, input and output; backward twice that; features,
        # target, weighted graph and three hidden fields in 16 bits, read and written once
        flops = 3 * 2 * n * (16 * 64 + 3 * 128 * 64 + 64 * 3)
        return dict(bytes=n * (32 + 12 + 8 * entries + 3 * 128), flops=flops)
    return _step_work(n, entries, case["precision"], case["steps"])


def _member_nodes(i):
    r = synth.uniform01(synth.substream(100 + i, 4), np.arange(1))[0]
    return 2000.0 * 100.0 ** r


# ------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------

_HEX_SIGN = torch.tensor([[-1, -1, -1], [1, -1, -1], [1, 1, -1], [-1, 1, -1], [-1, -1, 1],
                          [1, -1, 1], [1, 1, 1], [-1, 1, 1]], dtype=torch.float64)


class _Exact:
    """Finite elements of one periodic lattice mesh and the step's equations, FP64 torch."""

    def __init__(self, mesh, mat, dt=1e-12, alpha=0.5):
        dev, dt64 = "cuda", torch.float64
        nx, ny, nz = mesh.n_cells
        s = torch.arange(mesh.coords.shape[0], device=dev)
        i, j, k = s % (nx + 1), s // (nx + 1) % (ny + 1), s // ((nx + 1) * (ny + 1))
        node = i % nx + nx * (j % ny + ny * (k % nz))
        t = torch.as_tensor(mesh.tets.astype(np.int64), device=dev)
        x = torch.as_tensor(mesh.coords, device=dev)[t]                    # [e, k, 3]
        self.t, self.n, self.nen = node[t], nx * ny * nz, t.shape[1]
        if self.nen == 4:
            J = x[:, 1:] - x[:, :1]                                       # rows: edges
            det = torch.linalg.det(J)
            inv = torch.linalg.inv(J)                                     # d xi / d x
            g = torch.cat([-inv.sum(2, keepdim=True), inv], 2).transpose(1, 2)
            self.G, self.w = g[:, None], (det / 6.0)[:, None]             # one point
            self.N = torch.full((1, 4), 0.25, device=dev, dtype=dt64)
            Me = (torch.ones(4, 4, device=dev, dtype=dt64) + torch.eye(4, device=dev)) / 20.0
            self.Me = self.w[:, :, None] * Me
        else:
            sg = _HEX_SIGN.to(dev)
            xi = sg / math.sqrt(3.0)
            f = 1.0 + xi[:, None, :] * sg[None]                           # [q, k, 3]
            self.N = f.prod(2) / 8.0
            d = torch.stack([sg[None, :, a] * f[..., (a + 1) % 3] * f[..., (a + 2) % 3]
                             for a in range(3)], 2) / 8.0                 # [q, k, 3]
            J = torch.einsum("qka,ekb->eqab", d, x)                       # d x_b / d xi_a
            self.w = torch.linalg.det(J)
            self.G = torch.einsum("eqba,qka->eqkb", torch.linalg.inv(J), d)
            self.Me = torch.einsum("eq,qk,ql->ekl", self.w, self.N, self.N)
        self.V = self.w.sum(1)
        self.ML = torch.zeros(self.n, device=dev, dtype=dt64)
        self.ML.index_add_(0, self.t.reshape(-1), (self.w @ self.N).reshape(-1))
        self.volume = self.V.sum()
        em = torch.as_tensor(mesh.elem_magnetic.astype(bool), device=dev)
        self.em = em
        self.mag = torch.zeros(self.n, dtype=torch.bool, device=dev)
        self.mag[self.t[em].reshape(-1)] = True
        # reduced constants
        self.mat = mat
        sc = MU0 * mat["Ms"] ** 2
        self.kappa = 2.0 * mat["K1"] / sc
        self.dtau, self.alpha = GAMMA0 * mat["Ms"] * dt, alpha
        self.eps = 2.0 * mat["A"] / (sc * 1e-18) * self.dtau
        self.me = 3.0 / sc
        self.Nd = torch.tensor(mat["Nd"], device=dev, dtype=dt64).reshape(3, 3)
        C = torch.zeros(3, 3, 3, 3, dtype=dt64)
        for a in range(3):
            C[a, a, a, a] = mat["C11"]
            for b in range(3):
                if a != b:
                    C[a, a, b, b] = mat["C12"]
                    C[a, b, a, b] = C[a, b, b, a] = mat["C44"]
        self.C = C.to(dev)

    def csr(self, blocks, sel=None):
        """Element blocks [e, k, a, k, b] summed into a sparse matrix (nodes x components)."""
        t = self.t if sel is None else self.t[sel]
        nc = blocks.shape[2]
        dof = (nc * t[:, :, None] + torch.arange(nc, device=t.device)).reshape(t.shape[0], -1)
        m = dof.shape[1]
        idx = torch.stack([dof[:, :, None].expand(-1, m, m).reshape(-1),
                           dof[:, None, :].expand(-1, m, m).reshape(-1)])
        A = torch.sparse_coo_tensor(idx, blocks.reshape(-1), (nc * self.n, nc * self.n))
        return A.coalesce().to_sparse_csr()

    def scalar(self, el, sel=None):
        return self.csr(el[:, :, None, :, None], sel)

    def build(self):
        Ke = torch.einsum("eq,eqka,eqla->ekl", self.w, self.G, self.G)
        self.Kms = self.scalar(Ke)
        self.F = [self.scalar(-torch.einsum("eq,qk,eql->ekl", self.w, self.N, self.G[..., a]))
                  for a in range(3)]
        self.Kmech = self.csr(torch.einsum("eq,eqkc,acbd,eqld->ekalb", self.w, self.G, self.C,
                                           self.G))
        Km, Mm = Ke[self.em], self.Me[self.em]
        self.Mgs = self.scalar(Mm, self.em)
        self.Ae = self.scalar(Mm + self.eps * Km, self.em)
        self.Aa = self.scalar(Mm + self.alpha * self.eps * Km, self.em)
        return self

    @staticmethod
    def cg(A, b, x, diag, project=None):
        r = b - A @ x
        if project is not None:
            r = project(r)
        z = r / diag if project is None else project(r / diag)
        p, rz, bb = z.clone(), r @ z, float(b @ b)
        for it in range(20000):
            q = A @ p
            al = rz / (p @ q)
            x = x + al * p
            r = r - al * q
            if it % 8 == 7 and float(r @ r) < 1e-24 * bb:
                break
            z = r / diag if project is None else project(r / diag)
            rz, old = r @ z, rz
            p = z + (rz / old) * p
        return x

    def diagonal(self, A):
        crow, col, val = A.crow_indices(), A.col_indices(), A.values()
        row = torch.repeat_interleave(torch.arange(A.shape[0], device=val.device),
                                      crow[1:] - crow[:-1])
        d = torch.ones(A.shape[0], device=val.device, dtype=val.dtype)
        on = row == col
        d[row[on]] = val[on]
        return d

    def singular(self, A, b, nc):
        """K x = b on the periodic mesh, shifted to zero at node 0."""
        if not float(b.abs().max()) > 0.0:
            return torch.zeros_like(b)
        proj = lambda v: (v.reshape(-1, nc) - v.reshape(-1, nc).mean(0)).reshape(-1)  # noqa: E731
        b = proj(b)
        x = self.cg(A, b, torch.zeros_like(b), self.diagonal(A), proj).reshape(-1, nc)
        return (x - x[:1]).reshape(-1)

    def mean(self, f):
        return torch.tensordot(self.ML, f, dims=1) / self.volume

    def strain0(self, m):
        E = 1.5 * self.mat["lambda111"] * m[:, :, None] * m[:, None, :]
        for a in range(3):
            E[:, a, a] = 1.5 * self.mat["lambda100"] * (m[:, a] ** 2 - 1.0 / 3.0)
        E[~self.mag] = 0.0
        return E

    def stress(self, E):
        return torch.einsum("abcd,ncd->nab", self.C, E)

    def elastic(self, m):
        E0 = self.strain0(m)
        S = self.stress(E0)[self.t]                                       # [e, k, 3, 3]
        el = torch.einsum("eq,eqkc,ql,elac->eka", self.w, self.G, self.N, S)
        b = torch.zeros(self.n, 3, device=m.device, dtype=m.dtype)
        b.index_add_(0, self.t.reshape(-1), el.reshape(-1, 3))
        u = self.singular(self.Kmech, b.reshape(-1), 3).reshape(-1, 3)
        return u, E0

    def gradient(self, v):
        return torch.stack([-(F @ v) / self.ML for F in self.F], 1)

    def field(self, m, hd, E, H):
        s = self.stress(E - self.strain0(m))
        l1, l4 = self.mat["lambda100"], self.mat["lambda111"]
        h = torch.empty_like(m)
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            h[:, a] = (-self.kappa * m[:, a] * (m[:, b] ** 2 + m[:, c] ** 2) + self.me *
                       (l1 * m[:, a] * s[:, a, a] + l4 * (m[:, b] * s[:, a, b] +
                                                          m[:, c] * s[:, a, c])))
        h = h + H + hd - self.Nd @ self.mean(m)
        h[~self.mag] = 0.0
        return h

    def smooth(self, A, diag, f):
        """(M + c eps K) g = M f on the magnetic nodes, zero elsewhere."""
        f = torch.where(self.mag, f, torch.zeros_like(f))
        return self.cg(A, self.Mgs @ f, f, diag)

    def step(self, m, H):
        b = sum(F @ m[:, a].contiguous() for a, F in enumerate(self.F))
        U = self.singular(self.Kms, b, 1)
        hd = -self.gradient(U)
        u, E0 = self.elastic(m)
        Du = torch.stack([self.gradient(u[:, b].contiguous()) for b in range(3)], 1)
        E = self.mean(E0) + 0.5 * (Du + Du.transpose(1, 2))
        h = self.field(m, hd, E, H)
        de, da, dt = self.diagonal(self.Ae), self.diagonal(self.Aa), self.dtau
        g2 = self.smooth(self.Ae, de, m[:, 1] + dt * h[:, 1])
        g3 = self.smooth(self.Ae, de, m[:, 2] + dt * h[:, 2])
        s1 = m[:, 0] + (g2 * m[:, 2] - g3 * m[:, 1])
        g1 = self.smooth(self.Ae, de, s1 + dt * h[:, 0])
        s2 = m[:, 1] + (g3 * s1 - g1 * m[:, 2])
        g2 = self.smooth(self.Ae, de, s2 + dt * h[:, 1])
        s3 = m[:, 2] + (g1 * s2 - g2 * s1)
        ms = torch.stack([s1, s2, s3], 1)
        ms[~self.mag] = 0.0
        f = ms + self.alpha * dt * self.field(ms, hd, E, H)
        x = torch.stack([self.smooth(self.Aa, da, f[:, a]) for a in range(3)], 1)
        out = torch.zeros_like(m)
        out[self.mag] = x[self.mag] / x[self.mag].norm(dim=1, keepdim=True)
        return out, U, u

    def steps(self, m, H, steps):
        m = torch.where(self.mag[:, None], m, torch.zeros_like(m))
        H = torch.tensor(H, device=m.device, dtype=m.dtype) / self.mat["Ms"]
        for _ in range(steps):
            m, U, u = self.step(m, H)
        return m, U, u

    def loss_and_gradient(self, flat, m, u1, u0, target):
        """Loss and gradients of the warm-start network (see gspm_mpnn_* in include/gspm.h)."""
        k = self.nen
        B = self.scalar((self.V / k)[:, None, None].expand(-1, k, k))
        rows = B @ torch.ones(self.n, device=m.device, dtype=m.dtype)
        l1, l4 = self.mat["lambda100"], self.mat["lambda111"]
        ls = max(abs(l1), abs(l4))
        us = ls * float((self.volume / self.n) ** (1.0 / 3.0))
        m = torch.where(self.mag[:, None], m, torch.zeros_like(m))
        E = self.strain0(m)
        ev = torch.stack([E[:, 0, 0], E[:, 1, 1], E[:, 2, 2], E[:, 1, 2], E[:, 0, 2],
                          E[:, 0, 1]], 1) / ls
        f = torch.cat([m, ev, u1 / us, (u1 - u0) / us, torch.ones_like(m[:, :1])], 1)
        par = torch.as_tensor(flat, dtype=torch.float64, device=m.device).requires_grad_(True)
        p, o = {}, 0
        for key, shape in gspm.MPNN_KEYS:
            size = int(np.prod(shape))
            p[key] = par[o:o + size].reshape(shape)
            o += size
        h = torch.relu(f @ p["W_in"] + p["b_in"])
        for layer in (1, 2, 3):
            z = torch.sparse.mm(B, h) / rows[:, None]
            h = torch.relu(torch.cat([h, z], 1) @ p["W%d" % layer] + p["b%d" % layer])
        y = h @ p["W_out"] + p["b_out"]
        loss = ((y - (target - (2 * u1 - u0)) / us) ** 2).mean()
        loss.backward()
        return float(loss.detach()), par.grad


def exact(case, seed):
    kind = case["kind"]
    state = {}
    if kind == "average_noalloc":
        state = prepare(case, seed)
        return torch.tensordot(state["weights"], state["field"], dims=1)
    gen = _generator(seed)
    if kind == "batch":
        cfgs = _batch_configs(case["first"], case["count"])
        if sum(c["mesh"].n_unique for c in cfgs) > EXACT_NODES:
            return None
        parts = []
        for c in cfgs:
            m = _magnetisation(c["mesh"].n_cells, gen)
            fe = _Exact(c["mesh"], c["material"], c["dt"], c["alpha"]).build()
            parts.append(fe.steps(m, c["H"], case["steps"]))
        return dict(zip(("m", "U", "u"), (torch.cat(v) for v in zip(*parts))))
    sides = _sides(case)
    n = sides[0] * sides[1] * sides[2]
    mesh, mat = _mesh(case["cells"], case["recipe"])
    if kind == "average":
        f = 0.5 + torch.randn(n, case["ncomp"], generator=gen, device="cuda", dtype=torch.float64)
        return _Exact(mesh, mat).mean(f).cpu().numpy()
    if n > (3 * EXACT_NODES if kind == "elastic" else EXACT_NODES):
        return None
    m = _magnetisation(sides, gen)
    if kind == "elastic":
        fe = _Exact(mesh, mat)
        fe.Kmech = fe.csr(torch.einsum("eq,eqkc,acbd,eqld->ekalb", fe.w, fe.G, fe.C, fe.G))
        return fe.elastic(torch.where(fe.mag[:, None], m, torch.zeros_like(m)))[0]
    if kind == "grad":
        u1 = _displacement(sides, gen)
        u0 = u1 + 0.1 * _displacement(sides, gen)
        target = u1 + 0.1 * _displacement(sides, gen)
        loss, grad = _Exact(mesh, mat).loss_and_gradient(_weights(), m, u1, u0, target)
        return dict(loss=loss, grad=grad)
    fe = _Exact(mesh, mat, case["dt"], case["alpha"]).build()
    return dict(zip(("m", "U", "u"), fe.steps(m, [case["field_T"] / MU0, 0.0, 0.0],
                                              case["steps"])))
