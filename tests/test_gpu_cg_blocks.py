"""The cooperative approximate-Jacobian solve at the sizes where its launch
changes: fewer cells than a block, one block exactly, one cell more, and more
cells than one a thread on every SM (the kernel that walks its cells), with
3 to 16 face slots a cell, against Jacobi-preconditioned conjugate gradients
in numpy on the matrix the library reports.

Bars after 12 iterations: FP64 1e-11 (12 iterations' rounding of sums over
the cells, ~1e-15 each, through the recurrences), FP32 1e-4 (the same with
2^-24)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2601_18417_gb300 import hofv
from paper_2601_18417_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ITERS = 12
SIZES = [("tensor", 2, 9), ("tensor", 2, 32), ("tensor", 3, 12), ("simplex", 2, 23),
         ("simplex", 3, 6), ("polygon", 2, 32), ("polyhedron", 3, 9), ("tensor", 2, 400),
         ("tensor", 3, 55)]


def _cg(diag, a, b, off, v, kbar):
    x, r = np.zeros_like(v), -v / kbar

    def mul(p):
        y = -diag * p
        for j in range(p.shape[0]):
            y[j] -= np.bincount(a, off * p[j, b], p.shape[1]) + np.bincount(b, off * p[j, a], p.shape[1])
        return y
    z = r / -diag
    p, rz = z.copy(), (r * z).sum(1, keepdims=True)
    for _ in range(ITERS):
        q = mul(p)
        al = rz / (p * q).sum(1, keepdims=True)
        x, r = x + al * p, r - al * q
        z = r / -diag
        new = (r * z).sum(1, keepdims=True)
        p, rz = z + new / rz * p, new
    return x


@pytest.mark.parametrize("kind,dim,n", SIZES)
def test_cooperative_cg_against_numpy(kind, dim, n):
    import torch
    mesh = I.make_mesh(dim, n, jitter=0.1, seed=2, cells=kind)
    if hasattr(mesh, "face_ptr"):
        tags = np.where(mesh.face_side >= 0, 0, -1).astype(np.int32)
    else:
        tags = np.zeros(mesh.bface_side.size, np.int32)
    ctx = hofv.Context(0)
    ctx.set_mesh(mesh, tags)
    ctx.set_scheme(1, 10 if dim == 2 else 20, 1)
    lay = ctx.build_stencils()
    ctx.set_material(hofv.LAW_LINEAR, 1.0, 1.5)
    diag, off = ctx.get_aj()
    own, nei, _, _ = ctx.get_faces()
    m = lay.n_internal
    v = np.random.default_rng(4).standard_normal((dim, lay.n_cells))
    ref = _cg(diag, own[:m], nei[:m], off, v, 3.5)
    vd = torch.as_tensor(v, device="cuda:0")
    for pc, bar in ((hofv.PC_AJ64, 1e-11), (hofv.PC_AJ32, 1e-4)):
        z = torch.full_like(vd, float("nan"))
        ctx.precondition(pc, ITERS, vd, z)
        first = z.clone()
        ctx.precondition(pc, ITERS, vd, z)
        assert torch.equal(z, first)  # the barrier's counters are clear again
        err = np.linalg.norm(z.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= bar, (pc, err)
    ctx.close()
