"""The default precision on states whose values differ by orders of magnitude
within a stencil: a column of the operator (one cell, one component set), one
value a million times its neighbours, a field falling by ten a cell.

Every cell's residual is held to the bound of FP64 sums, (S + 20) 2^-53 times
the sum of the magnitudes of all the terms that enter it (S for a sum over a
stencil, the rest for the products of the law, the quadrature and the
assembly; the prefactor 2 for the difference of extrapolated values), against
the same sums in extended precision from the coefficients the library
reports."""
from __future__ import annotations

import numpy as np
import pytest

from tests import helpers as H
from tests.test_gpu_polyhedra import _context as polyhedral_context

pytestmark = pytest.mark.gpu
LD = np.longdouble
MU, LAM, ALPHA = 1.0, 1.5, 0.1


def _reference(ctx, pb, u, absolute):
    """R(u) of the linear law without data, or the sum of its terms' magnitudes."""
    o, d = pb.orc, pb.dim
    mag = (lambda x: np.abs(x).astype(LD)) if absolute else (lambda x: x.astype(LD))
    nf = ctx.layout.n_internal + ctx.layout.n_disp
    st, co = ctx.get_face_data(0, nf)
    cst, ex = ctx.get_cell_data(0, o.nc)
    a = mag(o.aq[:nf, :, :d])  # the library's polyhedral faces may have more points, without area
    co, ex, uu = mag(co[:, :a.shape[1], :-1]), mag(ex), mag(u)
    G = np.zeros((nf, co.shape[1], d, d), LD)
    us = np.repeat(uu.T[:, None, :], ex.shape[1], axis=1)
    for n in range(st.shape[1]):  # a slot at a time
        G += co[:, :, n, :, None] * uu[:, st[:, n]].T[:, None, None, :]
        us += ex[:, :, n, None] * uu[:, cst[:, n]].T[:, None, :]
    T = MU * (np.einsum("fqij,fqj->fi", G, a) + np.einsum("fqji,fqj->fi", G, a)) \
        + LAM * np.einsum("fqkk,fqi->fi", G, a)
    own, nei, _, _ = ctx.get_faces()
    own, nei = own[:nf], nei[:nf]
    slot = {(c, f): lf for c, row in enumerate(o.cell_faces()) for lf, f in enumerate(row)}
    up = np.stack([us[own[f], slot[own[f], f]] for f in range(nf)])
    un = np.stack([us[nei[f], slot[nei[f], f]] if nei[f] >= 0 else np.zeros(d, LD) for f in range(nf)])
    dx = np.where((nei >= 0)[:, None], o.xc[np.maximum(nei, 0)], o.xf[:nf]) - o.xc[own]
    w = ALPHA * (2 * MU + LAM) * o.gamma[:nf] / np.abs((dx * o.normal[:nf]).sum(1))
    flux = T + w[:, None] * (un + up if absolute else un - up)
    R = np.zeros((d, o.nc), LD)
    for f in range(nf):
        R[:, own[f]] += flux[f]
        if nei[f] >= 0:
            R[:, nei[f]] += flux[f] if absolute else -flux[f]
    return R


@pytest.mark.parametrize("dim,n,p,q1,kind", [(2, 12, 2, 2, "tensor"), (2, 11, 3, 3, "tensor"),
                                             (2, 8, 3, 2, "simplex"), (3, 6, 2, 2, "tensor"),
                                             (3, 6, 3, 3, "tensor"), (3, 5, 1, 1, "tensor"),
                                             (3, 4, 1, 1, "simplex"), (3, 4, 2, 2, "simplex"),
                                             (3, 5, 2, 2, "polyhedron")])
def test_terms_of_very_different_size(dim, n, p, q1, kind):
    import torch
    pb = H.make_problem(dim, n, p, q1, jitter=0.15, seed=3, kind=kind, alpha=ALPHA)
    # boundary data at the library's points, which may be more than the oracle's
    ctx = polyhedral_context(pb) if kind == "polyhedron" else H.gpu_context(pb)
    g, nc = np.random.default_rng(7), pb.orc.nc
    states = []
    for cell in (nc // 2, int(g.integers(nc))):
        u = np.zeros((dim, nc))
        u[g.integers(dim), cell] = 1.1
        states.append(u)
    u = g.standard_normal((dim, nc))
    u[:, nc // 3] *= 1e6
    states.append(u)
    direction = g.standard_normal(dim)
    s = pb.orc.xc[:, :dim] @ (direction / np.linalg.norm(direction)) * n
    states.append((1.0 + g.random((dim, 1))) * 10.0 ** -s)
    bar = 2.0 * (ctx.layout.stencil + 20) * 2.0 ** -53
    for k, u in enumerate(states):
        ud = H.to_dev(u)
        R = torch.empty_like(ud)
        ctx.residual(ud, R)
        err = np.abs(R.cpu().numpy() - _reference(ctx, pb, u, False))
        assert (err <= bar * _reference(ctx, pb, u, True)).all(), k
    ctx.close()
