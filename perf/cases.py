"""The work that a user of this library has it do, as cases to be timed.

A case is one call of the public binding (`hofv.Context`) on one mesh: a
residual, a Jacobian-vector product, a flexible Arnoldi step (preconditioner,
product, orthogonalisation), one application of the preconditioner, or a whole
Newton-Krylov solve.  Meshes, orders and materials are those of the workloads
in `paper_2601_18417_gb300/inputs.py` and of the tests, at sizes whose set-up
takes seconds; states are smooth fields with noise, as in `bench.py`.

`exact` evaluates the same discretisation in 64-bit torch from the paper's
equations (arXiv 2601.18417; the readings are those of the library's header).
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

from paper_2601_18417_gb300 import hofv
from paper_2601_18417_gb300 import inputs as I

E_MOD, NU = 1e9, 0.3            # linear cases (hex96-p3-trig)
MU_NH, LAM_NH = 1e6, 4e6        # the neo-Hookean block
ALPHA, K_WEIGHT = 0.1, 6.0
PC = {"AJ32": hofv.PC_AJ32, "AJMG": hofv.PC_AJMG}


def _case(name, call, cells, dim, n, p, law="linear", precision="fp64", contracted=False, pc="",
          inner=0, basis=0, jitter=0.2):
    return {"name": name, "call": call, "cells": cells, "dim": dim, "n": n, "p": p, "law": law,
            "precision": precision, "contracted": contracted, "pc": pc, "inner": inner,
            "basis": basis, "jitter": jitter}


def listed():
    return [
        # the smallest whole call: quad32-p2-trig solved with the library's default options
        # (FP64 contraction, 30 FP32 Jacobi-CG iterations a preconditioning)
        _case("newton_quad32_p2", "newton", "tensor", 2, 32, 2, pc="AJ32", inner=30, jitter=0.0),
        # a small neo-Hookean block to its first load step with the multigrid inner solve
        _case("newton_hex12_p2_nh", "newton", "tensor", 3, 12, 2, "neo-hookean", "df64",
              pc="AJMG", inner=1),
        # the smallest single call: one product on an odd-sized block, latency counts
        _case("jvp_hex13_p3_nh", "jvp", "tensor", 3, 13, 3, "neo-hookean", "df64"),
        # quad512j-p3-mixed: the step the solver repeats, 16 basis vectors
        _case("arnoldi_quad512_p3", "arnoldi", "tensor", 2, 512, 3, precision="df64", pc="AJMG",
              inner=1, basis=16, jitter=0.25),
        # the same mesh, Hooke's law folded into the coefficients (hofv_set_contraction)
        _case("residual_quad512_p3_contracted", "residual", "tensor", 2, 512, 3, contracted=True,
              jitter=0.25),
        # unstructured triangles in the library's default arithmetic
        _case("residual_tri255_p3_fp64", "residual", "simplex", 2, 255, 3, jitter=0.15),
        # the block of the load-step comparison (hex64j-p2-nh): one step of its solver
        _case("arnoldi_hex64_p2_nh", "arnoldi", "tensor", 3, 64, 2, "neo-hookean", "df64",
              pc="AJMG", inner=1, basis=16),
        # the benchmark's scheme (hex128j-p3-nh) at the size that fits three times over
        _case("arnoldi_hex64_p3_nh", "arnoldi", "tensor", 3, 64, 3, "neo-hookean", "df64",
              pc="AJMG", inner=1, basis=16),
        # hex32j-p3-nh in the default arithmetic
        _case("residual_hex32_p3_nh_fp64", "residual", "tensor", 3, 32, 3, "neo-hookean"),
        # polyhedra given face by face (prism24j-p2-trig)
        _case("jvp_prism24_p2", "jvp", "polyhedron", 3, 24, 2, precision="df64", jitter=0.1),
        # unstructured tetrahedra (tet32j-p2-trig's scheme)
        _case("jvp_tet17_p2", "jvp", "simplex", 3, 17, 2, precision="df64", jitter=0.1),
        # the default preconditioner alone on the paper's 45^3 grid
        _case("precondition_hex45_aj32", "precondition", "tensor", 3, 45, 1, pc="AJ32", inner=30),
    ]


# range of sizes of each listed kind; the other fields are the listed case's
_RANGES = {"newton_quad32_p2": (14, 64), "newton_hex12_p2_nh": (6, 13), "jvp_hex13_p3_nh": (8, 45),
           "arnoldi_quad512_p3": (60, 512), "residual_quad512_p3_contracted": (60, 512),
           "residual_tri255_p3_fp64": (40, 300), "arnoldi_hex64_p2_nh": (14, 64),
           "arnoldi_hex64_p3_nh": (16, 56), "residual_hex32_p3_nh_fp64": (8, 33),
           "jvp_prism24_p2": (7, 24), "jvp_tet17_p2": (5, 20), "precondition_hex45_aj32": (12, 52)}


def draw(rng):
    """One more case: a listed kind at a size spread over its range on a
    logarithmic scale, with the order, law and precision it may also have."""
    c = dict(rng.choice(listed()))
    lo, hi = _RANGES[c.pop("name")]
    c["n"] = min(hi, int(round(lo * (hi / lo) ** rng.random())))
    if c["call"] != "newton":
        c["jitter"] = rng.choice([0.05, 0.1, 0.15]) if c["cells"] != "tensor" else rng.choice([0.1, 0.2])
    if c["dim"] == 2 and c["call"] != "newton":
        c["p"] = rng.choice([2, 3])
        if not c["contracted"]:
            c["precision"] = rng.choice(["fp64", "df64"]) if c["call"] == "residual" else "df64"
    if c["call"] == "jvp" and c["cells"] == "tensor":
        c["law"] = rng.choice(["linear", "neo-hookean"])
    if c["basis"]:
        c["basis"] = rng.randrange(1, 25)
    if c["call"] == "precondition":
        c["inner"] = rng.randrange(10, 31)
    return c


# ---------------------------------------------------------------- the problem
def _n_plus(case):
    return 10 if case["dim"] == 2 else {1: 45, 2: 55, 3: 65}[case["p"]]


def _stencil(case):
    return math.comb(case["dim"] + case["p"], case["dim"]) + _n_plus(case)


def _q1(case):
    return 3 if case["p"] == 3 else 2


def _moduli(case):
    return I.lame_from_young(E_MOD, NU) if case["law"] == "linear" else (MU_NH, LAM_NH)


def _mesh(case, seed):
    """The mesh and one boundary tag per domain side (0 displacement, 1 traction)."""
    mesh = I.make_mesh(case["dim"], case["n"], jitter=case["jitter"], seed=seed, cells=case["cells"])
    return mesh, I.side_tags("block" if case["law"] == "neo-hookean" else "mms", case["dim"])


def _waves(dim, seed):
    """Amplitudes, wave vectors and phases of the seeded displacement field."""
    g = np.random.default_rng([seed, 17])
    return (1e-3 * (1.0 + g.random((3, dim))), 2.0 * math.pi * (0.5 + g.random((3, dim))),
            2.0 * math.pi * g.random((3, dim)))


def _field(case, seed, x):
    """Displacement at the points x [..., dim]: three seeded waves (linear law),
    or the block pushed down by 3 % of its height (its first load step)."""
    dim = case["dim"]
    if case["law"] == "neo-hookean":
        u = torch.zeros_like(x)
        u[..., dim - 1] = -0.03 * x[..., dim - 1]
        return u
    a, k, ph = (torch.as_tensor(t, dtype=x.dtype, device=x.device) for t in _waves(dim, seed))
    s = torch.sin(torch.einsum("...i,wi->...w", x, k)[..., None] + ph)
    return (a * s).sum(-2)


def _prescribed(case, seed, x):
    """Prescribed displacement at boundary points x [..., dim]."""
    if case["law"] == "neo-hookean":
        u = torch.zeros_like(x)
        u[..., -1] = torch.where(x[..., -1] > 0.5, -0.03, 0.0)
        return u
    return _field(case, seed, x)


def _body(case, seed, xc, vol):
    """Body force of each cell [dim, nc]: a seeded smooth load times the volume."""
    dim, mu = case["dim"], _moduli(case)[0]
    if case["law"] == "neo-hookean":
        b = torch.zeros_like(xc)
        b[:, -1] = -1e-3 * mu
    else:
        b = mu * 20.0 * _field(case, seed + 1, xc)
    return (b * vol[:, None]).T.contiguous()


def _random(case, seed, shape, stream):
    g = torch.Generator(device=_device()).manual_seed(1_000_003 * stream + seed)
    return torch.randn(shape, generator=g, dtype=torch.float64, device=_device())


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _state(case, seed, xc):
    """u [dim, nc]: the field at the centroids plus noise of 1e-3 of its largest value."""
    u = _field(case, seed, xc).T.contiguous()
    return u + 1e-3 * u.abs().max() * _random(case, seed, u.shape, 1)


def _direction(case, seed, nc):
    v = _random(case, seed, (case["dim"], nc), 2)
    return v / v.norm()


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    dim = case["dim"]
    mesh, side = _mesh(case, seed)
    if hasattr(mesh, "face_ptr"):
        tags = np.where(mesh.face_side >= 0, side[np.maximum(mesh.face_side, 0)], -1).astype(np.int32)
    else:
        tags = side[mesh.bface_side]
    ctx = hofv.Context(0)
    ctx.set_mesh(mesh, tags)
    ctx.set_scheme(case["p"], _n_plus(case), _q1(case), K_WEIGHT, ALPHA)
    ctx.set_precision(hofv.PREC_DF64 if case["precision"] == "df64" else hofv.PREC_FP64)
    lay = ctx.build_stencils()
    ctx.set_material(hofv.LAW_NEOHOOKEAN if case["law"] == "neo-hookean" else hofv.LAW_LINEAR,
                     *_moduli(case))
    if case["contracted"]:
        ctx.set_contraction(True)
    pts = lambda kind: torch.as_tensor(ctx.get_points(kind), device="cuda")  # noqa: E731
    xc = pts(hofv.PTS_CELL_CENTROID)
    ctx.set_bc(_prescribed(case, seed, pts(hofv.PTS_DISP_QP)).contiguous(),
               _prescribed(case, seed, pts(hofv.PTS_DISP_CENTRE)).contiguous(), None,
               _body(case, seed, xc, pts(hofv.PTS_CELL_VOLUME)))
    s = {"case": case, "ctx": ctx}
    if case["pc"] == "AJMG":
        ctx.mg_info()                       # the hierarchy, once per mesh
    if case["call"] == "newton":
        s["start"] = _field(case, seed, xc).T.contiguous() if case["law"] == "neo-hookean" \
            else torch.zeros((dim, lay.n_cells), dtype=torch.float64, device="cuda")
        s["u"] = s["start"].clone()
        ctx.prepare_solver(precond=PC[case["pc"]], inner_iters=case["inner"])
        return s
    s["u"] = _state(case, seed, xc)
    s["R"] = torch.empty_like(s["u"])
    if case["call"] in ("jvp", "arnoldi"):
        ctx.residual(s["u"], s["R"])
    if case["call"] in ("jvp", "precondition"):
        s["v"] = _direction(case, seed, lay.n_cells)
        s["out"] = torch.empty_like(s["u"])
    if case["call"] == "arnoldi":
        k = case["basis"]
        s["V"] = _random(case, seed, (k + 1, dim * lay.n_cells), 3)
        s["V"] /= s["V"].norm(dim=1, keepdim=True)
        s["Z"] = torch.zeros_like(s["V"])
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["call"] == "newton":
        s["u"].copy_(s["start"])
        ctx.newton_solve(s["u"], precond=PC[case["pc"]], inner_iters=case["inner"])
        return s["u"]
    if case["call"] == "residual":
        ctx.residual(s["u"], s["R"])
        return s["R"]
    if case["call"] == "jvp":
        ctx.jvp(s["u"], s["R"], s["v"], s["out"])
        return s["out"]
    if case["call"] == "precondition":
        ctx.precondition(PC[case["pc"]], case["inner"], s["v"], s["out"])
        return s["out"]
    j = case["basis"] - 1
    h = ctx.arnoldi_step(s["u"], s["R"], PC[case["pc"]], case["inner"], s["V"], s["Z"], j)
    return [h, s["V"][j + 1], s["Z"][j]]


# ------------------------------------------------------------------- the work
def _counts(case):
    """(cells, faces with a flux, Gauss points with area on them, faces of a cell)."""
    n, d, q = case["n"], case["dim"], _q1(case)
    if case["cells"] == "polyhedron":
        # (n+1)^2 dual polygons of 2 n^2 triangles, n layers; a corner is q^2 points
        inner, rim = 3 * n * n + 2 * n, 8 * n
        level, sides = (n + 1) ** 2, inner + rim
        corners = (n + 1) * (2 * inner + rim) + 4 * n * sides
        faces = (n + 1) * level + n * sides
        return level * n, faces, corners * q * q, 2.0 * faces / (level * n)
    if case["cells"] == "simplex":
        nc = 2 * n * n if d == 2 else 6 * n ** 3
        faces = 3 * n * n + 2 * n if d == 2 else 12 * n ** 3 + 6 * n * n
        return nc, faces, faces * q ** (d - 1), d + 1
    faces = d * (n + 1) * n ** (d - 1)
    if case["law"] == "neo-hookean":      # traction-free sides carry no unknown flux
        faces -= 2 * (d - 1) * n ** (d - 1)
    return n ** d, faces, faces * q ** (d - 1), 2 * d


def work(case):
    """Bytes and operations of one call: coefficients, stencils, geometry and
    vectors once each.  A solve counts its Krylov iterations (about 60 on the
    32^2 quads, 8 on the small block), each a product and its vectors."""
    d, S = case["dim"], _stencil(case)
    nc, faces, points, nlf = _counts(case)
    vec = 8 * d * nc
    per_cell = 8 * nlf * S + 4 * S + 4 * nlf          # extrapolation weights, stencil, faces
    if case["contracted"]:
        face_b, face_f = faces * (8 * d * d * S + 4 * S + 16), 2.0 * faces * d * d * S
    else:
        face_b = points * (8 * d * S + 24) + faces * (4 * S + 16)
        face_f = points * (2.0 * d * d * S + (150 if case["law"] == "neo-hookean" else 6 * d * d))
    res_b = face_b + nc * per_cell + 2 * vec
    res_f = face_f + 2.0 * nc * nlf * S * d
    jv_b, jv_f = res_b + vec, res_f
    if case["law"] == "neo-hookean" and case["precision"] == "df64":
        jv_b += points * 8 * (d * d + d)              # the linearisation kept for the products
    if case["call"] == "residual":
        return {"bytes": res_b, "flops": res_f}
    if case["call"] == "jvp":
        return {"bytes": jv_b, "flops": jv_f}
    pc_b, pc_f = nc * (4 * nlf + 4 * nlf + 8) + 2 * vec, 4.0 * nc * nlf * d
    if case["call"] == "precondition":                # the operator is used once an iteration
        return {"bytes": pc_b, "flops": pc_f * case["inner"]}
    if case["call"] == "arnoldi":
        k = case["basis"]
        return {"bytes": pc_b + jv_b + (k + 2) * vec, "flops": pc_f + jv_f + 8.0 * k * d * nc}
    its = 60 if case["law"] == "linear" else 8
    return {"bytes": its * (jv_b + pc_b), "flops": its * (jv_f + pc_f * case["inner"])}


# ------------------------------------------------- the same in 64-bit torch
def exact(case, seed):
    if case["call"] == "arnoldi":        # holds a multigrid cycle: no closed value
        return None
    m = _Model(case, seed)
    if case["call"] == "residual":
        return m.residual(_state(case, seed, m.xc))
    if case["call"] == "jvp":
        return m.jvp(_state(case, seed, m.xc), _direction(case, seed, m.nc))
    if case["call"] == "precondition":
        return m.cg(_direction(case, seed, m.nc), case["inner"])
    return m.solve()


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w


def _patch(c, q):
    """Gauss points and vector areas of edges [F, 2, 2] or bilinear patches [F, 4, 3]."""
    gx, gw = _gauss(q)
    xs, aa = [], []
    if c.shape[-1] == 2:
        t = c[:, 1] - c[:, 0]
        for x, w in zip(gx, gw):
            xs.append((1 - x) * c[:, 0] + x * c[:, 1])
            aa.append(w * torch.stack([t[:, 1], -t[:, 0]], -1))
    else:
        for (x, w), (y, v) in itertools.product(zip(gx, gw), zip(gx, gw)):
            xs.append((1 - x) * (1 - y) * c[:, 0] + x * (1 - y) * c[:, 1] + x * y * c[:, 2]
                      + (1 - x) * y * c[:, 3])
            du = (1 - y) * (c[:, 1] - c[:, 0]) + y * (c[:, 2] - c[:, 3])
            dv = (1 - x) * (c[:, 3] - c[:, 0]) + x * (c[:, 2] - c[:, 1])
            aa.append(w * v * torch.cross(du, dv, dim=-1))
    return torch.stack(xs, 1), torch.stack(aa, 1)


_LOCAL = {("tensor", 2): ((3, 0), (1, 2), (0, 1), (2, 3)),
          ("tensor", 3): ((0, 4, 7, 3), (1, 2, 6, 5), (0, 1, 5, 4), (3, 7, 6, 2), (0, 3, 2, 1),
                          (4, 5, 6, 7)),
          ("simplex", 2): ((0, 1), (1, 2), (2, 0)),
          ("simplex", 3): ((0, 2, 1), (0, 1, 3), (0, 3, 2), (1, 2, 3))}


class _Model:
    """The scheme in 64 bits: faces with a flux (internal, then displacement)
    with Gauss points xq, vector areas aq, and the cells on both sides."""

    def __init__(self, case, seed):
        self.case, self.seed, self.dim, self.S = case, seed, case["dim"], _stencil(case)
        mesh, side = _mesh(case, seed)
        T = functools.partial(torch.as_tensor, device=_device())
        x = T(mesh.xyz)
        if hasattr(mesh, "face_ptr"):
            own, nei, tag = T(mesh.owner), T(mesh.neighbour), T(side.astype(np.int64))[
                T(np.maximum(mesh.face_side, 0).astype(np.int64))]
            xq, aq = self._fans(mesh, x, T)
        else:
            loc = np.array(_LOCAL[(case["cells"], self.dim)])
            fn = mesh.cell_nodes[:, loc]                             # [nc, faces, corners]
            flat = fn.reshape(-1, loc.shape[1])
            keys = np.sort(np.concatenate([flat, mesh.bface_nodes]), 1).astype(np.int64)
            key = keys[:, 0]
            for k in range(1, min(3, loc.shape[1])):                 # three corners fix a face
                key = key * mesh.n_nodes + keys[:, k]
            _, inv = np.unique(key, return_inverse=True)
            inv = inv.ravel()
            nslot, nf = flat.shape[0], int(inv.max()) + 1
            cell = np.arange(nslot) // loc.shape[0]
            first, last = np.full(nf, nslot), np.full(nf, -1)
            np.minimum.at(first, inv[:nslot], np.arange(nslot))
            np.maximum.at(last, inv[:nslot], np.arange(nslot))
            bside = np.full(nf, -1)
            bside[inv[nslot:]] = mesh.bface_side
            own, nei = T(cell[first]), T(np.where(first == last, -1, cell[last]))
            tag = T(side.astype(np.int64))[T(np.maximum(bside, 0))]
            corner = x[T(flat[first])]
            if corner.shape[1] == 3:
                corner = torch.cat([corner, corner[:, :1]], 1)
            xq, aq = _patch(corner, _q1(case))
        self.nc = mesh.n_cells
        inside = nei >= 0
        vol = torch.zeros(self.nc, dtype=x.dtype, device=x.device)
        mom = torch.zeros((self.nc, self.dim), dtype=x.dtype, device=x.device)
        for cells, sign, pick in ((own, 1.0, slice(None)), (nei[inside], -1.0, inside)):
            vol.index_add_(0, cells, sign * (xq * aq)[pick].sum((1, 2)) / self.dim)
            mom.index_add_(0, cells, sign * (xq * xq * aq)[pick].sum(1) / 2)
        self.vol, self.xc = vol, mom / vol[:, None]
        order = torch.cat([torch.nonzero(inside)[:, 0], torch.nonzero(~inside & (tag == 0))[:, 0]])
        self.ni = int(inside.sum())
        self.xq, self.aq, self.own, self.nei = xq[order], aq[order], own[order], nei[order[: self.ni]]
        mag = self.aq.norm(dim=-1)
        gam = mag.sum(1)
        self.xf = (mag[..., None] * self.xq).sum(1) / gam[:, None]
        nrm = torch.nn.functional.normalize(self.aq.sum(1), dim=1)
        far = torch.cat([self.xc[self.nei], self.xf[self.ni:]])
        self.stab = gam / ((far - self.xc[self.own]) * nrm).sum(1).abs()
        self.cut = x.amax(0) - x.amin(0)
        self.mu, self.lam = _moduli(case)
        self.ubq = _prescribed(case, seed, self.xq[self.ni:])
        self.ubf = _prescribed(case, seed, self.xf[self.ni:])
        self.body = _body(case, seed, self.xc, self.vol)

    def _fans(self, mesh, x, T):
        """Polyhedral faces: triangles from the corners' average, padded to the widest face."""
        q, deg = _q1(self.case), np.diff(mesh.face_ptr)
        width = int(deg.max())
        xq = torch.zeros((deg.size, width * q * q, 3), dtype=x.dtype, device=x.device)
        aq = torch.zeros_like(xq)
        for k in np.unique(deg):
            rows = np.nonzero(deg == k)[0]
            c = x[T(mesh.face_nodes[mesh.face_ptr[rows][:, None] + np.arange(k)])]
            mid, r = c.mean(1), T(rows)
            xq[r] = mid[:, None]
            for t in range(int(k)):
                a, b = _patch(torch.stack([mid, c[:, t], c[:, (t + 1) % int(k)], mid], 1), q)
                xq[r, t * q * q:(t + 1) * q * q] = a
                aq[r, t * q * q:(t + 1) * q * q] = b
        return xq, aq

    # ---- stencils: the S nearest centroids by the quantised squared distance, then by id
    def nearest(self, ref):
        d, nc, dev = self.dim, self.nc, ref.device
        e = math.floor(math.frexp(float(self.cut.prod()) / nc)[1] - 1)
        e = math.floor(e / d)
        scale, h = 2.0 ** (24 - 2 * e), 2.0 ** e
        lo = self.xc.amin(0)
        nb = ((self.xc.amax(0) - lo) / h).long() + 1
        mul = torch.cumprod(torch.cat([nb.new_ones(1), nb[:-1]]), 0)
        bucket = (((self.xc - lo) / h).long().clamp_(min=0) * mul).sum(1)
        ids = torch.argsort(bucket, stable=True)
        count = torch.bincount(bucket, minlength=int(nb.prod()))
        start = torch.cumsum(count, 0) - count
        cap = int(count.max())
        out = torch.empty((ref.shape[0], self.S), dtype=torch.int64, device=dev)
        todo, reach = torch.arange(ref.shape[0], device=dev), 3
        while todo.numel():
            off = torch.stack(torch.meshgrid(*[torch.arange(-reach, reach + 1, device=dev)] * d,
                                             indexing="ij"), -1).reshape(-1, d)
            left, step = [], max(1, 60_000_000 // (off.shape[0] * cap))
            whole = bool((nb <= reach).all())
            for part in torch.split(todo, step):
                r = ref[part]
                ib = torch.minimum(((r - lo) / h).floor().long().clamp_(min=0), nb - 1)
                k = ib[:, None] + off
                ok = ((k >= 0) & (k < nb)).all(-1)
                b = (torch.where(ok[..., None], k, 0) * mul).sum(-1)
                slot = torch.arange(cap, device=dev)
                has = ok[..., None] & (slot < count[b][..., None])
                cand = ids[torch.where(has, start[b][..., None] + slot, 0)]
                dx = self.xc[cand] - r[:, None, None]
                key = torch.floor((dx * dx).sum(-1) * scale + 0.5).long() * nc + cand
                key = torch.where(has, key, torch.iinfo(torch.int64).max).reshape(len(part), -1)
                n = min(self.S, key.shape[1])
                best = torch.topk(key, n, dim=1, largest=False).values
                edge = torch.minimum(torch.where(ib - reach > 0, r - (lo + (ib - reach) * h), 1e30),
                                     torch.where(ib + reach < nb - 1, lo + (ib + reach + 1) * h - r, 1e30))
                done = torch.full((len(part),), n == self.S, device=dev)
                done &= (best[:, -1] < torch.iinfo(torch.int64).max)
                if not whole:
                    done &= (best[:, -1] // nc + 2 < (edge.amin(1) ** 2 * scale))
                out[part[done]] = best[done] % nc if n == self.S else out[part[done]]
                left.append(part[~done])
            todo, reach = torch.cat(left), reach + 1
        return out

    def basis(self, X):
        cols, fact = [], (1.0, 1.0, 2.0, 6.0)
        for deg in range(self.case["p"] + 1):
            for a in range(deg, -1, -1):
                for b in ([deg - a] if self.dim == 2 else range(deg - a, -1, -1)):
                    t = X[..., 0] ** a * X[..., 1] ** b / (fact[a] * fact[b])
                    if self.dim == 3:
                        t = t * X[..., 2] ** (deg - a - b) / fact[deg - a - b]
                    cols.append(t)
        return torch.stack(cols, -1)

    def fit(self, ref, sten, ghost=False):
        """Weighted least squares at ref [B, dim] over sten [B, S]: (sqrt(w) Q [B, rows, Nt],
        R, h); a ghost row of weight 1 at ref where asked."""
        dx = self.xc[sten] - ref[:, None]
        r2 = (dx * dx).sum(-1)
        h = 2.0 * r2.amax(1).sqrt()
        X = dx / h[:, None, None]
        ek = math.exp(-K_WEIGHT ** 2)
        w = (torch.exp(-(X * X).sum(-1) * K_WEIGHT ** 2) - ek) / (1 - ek)
        A = self.basis(X)
        if ghost:
            row = torch.zeros_like(A[:, :1])
            row[..., 0] = 1.0
            A, w = torch.cat([A, row], 1), torch.cat([w, torch.ones_like(w[:, :1])], 1)
        sw = w.sqrt()[..., None]
        Q = A * sw
        nt = Q.shape[-1]
        R = torch.zeros((Q.shape[0], nt, nt), dtype=Q.dtype, device=Q.device)
        for k in range(nt):                              # Gram-Schmidt, twice
            v = Q[..., k]
            for _ in range(2 if k else 0):
                c = torch.einsum("brk,br->bk", Q[..., :k], v)
                v = v - torch.einsum("brk,bk->br", Q[..., :k], c)
                R[:, :k, k] += c
            R[:, k, k] = v.norm(dim=1)
            Q[..., k] = v / R[:, k, k, None]
        return Q * sw, R, h

    def _functional(self, fit, g):
        """Node weights [B, rows, m] of the functionals g [B, Nt, m]."""
        Q, R, _ = fit
        return Q @ torch.linalg.solve_triangular(R.transpose(1, 2), g, upper=False)

    def gradient_weights(self, chunk=1 << 21):
        """Yields (faces, points, stencils [B, S], weights [B, S(+1), dim]) over the face
        points with area; the last row is the ghost node of a displacement face."""
        sten = self.nearest(self.xf)
        f, q = torch.nonzero((self.aq != 0).any(-1), as_tuple=True)
        rows = max(1, chunk // (self.S * 4))
        for ghost, pick in ((False, f < self.ni), (True, f >= self.ni)):
            for ff, qq in zip(torch.split(f[pick], rows), torch.split(q[pick], rows)):
                if ff.numel() == 0:
                    continue
                fit = self.fit(self.xq[ff, qq], sten[ff], ghost)
                g = torch.zeros((ff.numel(), fit[1].shape[1], self.dim), dtype=torch.float64,
                                device=ff.device)
                for i in range(self.dim):
                    g[:, 1 + i, i] = 1.0 / fit[2]
                yield ff, qq, sten[ff], self._functional(fit, g)

    def sides(self):
        """(cell, face) of both sides of every face with a flux."""
        f = torch.arange(self.own.numel(), device=self.own.device)
        return torch.cat([self.own, self.nei]), torch.cat([f, f[: self.ni]])

    def side_weights(self, chunk=1 << 22):
        """Yields (side index, cells, stencils, weights [B, S]) of u* = u_P + sum e_N u_N."""
        cells, faces = self.sides()
        sten = self.nearest(self.xc)
        for k in torch.split(torch.arange(cells.numel(), device=cells.device), max(1, chunk // (self.S * 4))):
            c = cells[k]
            fit = self.fit(self.xc[c], sten[c])
            g = self.basis((self.xf[faces[k]] - self.xc[c]) / fit[2][:, None])
            g[:, 0] = 0.0
            yield k, c, sten[c], self._functional(fit, g[..., None])[..., 0]

    def traction(self, G, a):
        """t = T a from G[i][j] = du_j / dx_i."""
        if self.case["law"] == "linear":
            tr = G.diagonal(dim1=-2, dim2=-1).sum(-1)
            return self.mu * torch.einsum("...ij,...j->...i", G + G.transpose(-1, -2), a) \
                + self.lam * tr[..., None] * a
        F = G.transpose(-1, -2) + torch.eye(3, dtype=G.dtype, device=G.device)
        C, J = self._cofactor(F)
        B, w = F @ F.transpose(-1, -2), torch.einsum("...ij,...j->...i", C, a)
        trB = B.diagonal(dim1=-2, dim2=-1).sum(-1)
        kappa = self.lam + 2.0 * self.mu / 3.0
        iso = self.mu * J ** (-2.0 / 3.0)
        return ((iso / J)[..., None] * (torch.einsum("...ij,...j->...i", B, w) - trB[..., None] / 3 * w)
                + (0.5 * kappa * (J * J - 1) / J)[..., None] * w)

    @staticmethod
    def _cofactor(F):
        C = torch.stack([torch.cross(F[..., (i + 1) % 3, :], F[..., (i + 2) % 3, :], dim=-1)
                         for i in range(3)], -2)
        return C, (F[..., 0, :] * C[..., 0, :]).sum(-1)

    def traction_jvp(self, G, dG, a):
        """Derivative of the traction at G along dG."""
        if self.case["law"] == "linear":
            return self.traction(dG, a)
        return torch.func.jvp(lambda g: self.traction(g, a), (G,), (dG,))[1]

    def _assemble(self, flux):
        r = torch.zeros((self.nc, self.dim), dtype=flux.dtype, device=flux.device)
        r.index_add_(0, self.own, flux)
        r.index_add_(0, self.nei, -flux[: self.ni])
        return r

    def _evaluate(self, u, v=None):
        """Residual of u [dim, nc], or its derivative along v."""
        w = u.T.contiguous() if v is None else torch.cat([u, v]).T.contiguous()
        d = self.dim
        flux = torch.zeros((self.own.numel(), d), dtype=u.dtype, device=u.device)
        for f, q, sten, e in self.gradient_weights():
            G = torch.einsum("bni,bnj->bij", e[:, : self.S], w[sten])
            if e.shape[1] > self.S:
                G[..., :d] += e[:, self.S, :, None] * self.ubq[f - self.ni, q][:, None]
            a = self.aq[f, q]
            t = self.traction(G, a) if v is None else self.traction_jvp(G[..., :d], G[..., d:], a)
            flux.index_add_(0, f, t)
        w = w[:, -d:]
        star = torch.empty((self.own.numel() + self.ni, d), dtype=u.dtype, device=u.device)
        for k, c, sten, e in self.side_weights():
            star[k] = w[c] + torch.einsum("bn,bnj->bj", e, w[sten])
        nf = self.own.numel()
        other = torch.cat([star[nf:], self.ubf if v is None else torch.zeros_like(self.ubf)])
        flux += (ALPHA * (2 * self.mu + self.lam) * self.stab)[:, None] * (other - star[:nf])
        r = self._assemble(flux).T
        return (r + self.body if v is None else r).contiguous()

    def residual(self, u):
        return self._evaluate(u)

    def jvp(self, u, v):
        return self._evaluate(u, v)

    def cg(self, v, iters):
        """`iters` Jacobi-preconditioned CG iterations on the compact approximate Jacobian."""
        diag = torch.zeros(self.nc, dtype=v.dtype, device=v.device)
        diag.index_add_(0, self.own, self.stab)
        diag.index_add_(0, self.nei, self.stab[: self.ni])
        a, b, s = self.own[: self.ni], self.nei, self.stab[: self.ni]

        def mul(p):
            y = diag * p
            y.index_add_(1, a, -s * p[:, b])
            y.index_add_(1, b, -s * p[:, a])
            return y
        x, r = torch.zeros_like(v), -v / (2 * self.mu + self.lam)
        z = r / diag
        p, rz = z, (r * z).sum(1, keepdim=True)
        for _ in range(iters):
            q = mul(p)
            al = rz / (p * q).sum(1, keepdim=True)
            x, r = x + al * p, r - al * q
            z = r / diag
            new = (r * z).sum(1, keepdim=True)
            p, rz = z + new / rz * p, new
        return x

    def solve(self):
        """R(u) = 0 by Newton's method with the Jacobian as a dense matrix."""
        d, nc = self.dim, self.nc
        u = _field(self.case, self.seed, self.xc).T.contiguous() if self.case["law"] == "neo-hookean" \
            else torch.zeros((d, nc), dtype=torch.float64, device=self.xc.device)
        for it in range(12):
            R = self._evaluate(u)
            step = torch.linalg.solve(self._jacobian(u), -R.reshape(-1)).reshape(d, nc)
            u = u + step
            if step.norm() <= 1e-13 * u.norm() or self.case["law"] == "linear":
                break
        return u

    def _jacobian(self, u):
        d, nc, nf = self.dim, self.nc, self.own.numel()
        w = u.T.contiguous()
        J = torch.zeros((d * nc * d * nc,), dtype=u.dtype, device=u.device)

        def put(cells, cols, val):
            """J[i nc + cell, k nc + col] += val[..., i, k] for cells [B], cols [B, S]."""
            for i, k in itertools.product(range(d), range(d)):
                at = (i * nc + cells)[:, None] * (d * nc) + k * nc + cols
                J.index_add_(0, at.reshape(-1), val[..., i, k].reshape(-1))

        def both(f, cols, val):
            put(self.own[f], cols, val)
            m = f < self.ni
            put(self.nei[f[m]], cols[m], -val[m])
        for f, q, sten, e in self.gradient_weights():
            G = torch.einsum("bni,bnj->bij", e[:, : self.S], w[sten])
            if e.shape[1] > self.S:
                G += e[:, self.S, :, None] * self.ubq[f - self.ni, q][:, None]
            a, val = self.aq[f, q], torch.zeros((f.numel(), self.S, d, d), dtype=u.dtype, device=u.device)
            for i, k in itertools.product(range(d), range(d)):
                dG = torch.zeros_like(G)
                dG[:, i, k] = 1.0
                val[..., k] += e[:, : self.S, i, None] * self.traction_jvp(G, dG, a)[:, None]
            both(f, sten, val)
        eye = torch.eye(d, dtype=u.dtype, device=u.device)
        coef = ALPHA * (2 * self.mu + self.lam) * self.stab
        _, faces = self.sides()
        for k, c, sten, e in self.side_weights():
            f = faces[k]
            s = torch.where(k < nf, -coef[f], coef[f])
            cols, wts = torch.cat([c[:, None], sten], 1), torch.cat([torch.ones_like(e[:, :1]), e], 1)
            both(f, cols, (s[:, None] * wts)[..., None, None] * eye)
        return J.reshape(d * nc, d * nc)
