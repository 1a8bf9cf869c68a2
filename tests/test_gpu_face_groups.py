"""The double-float face and extrapolation kernels where their groups end:
face counts that are no multiple of a group (14, 16 or 32 faces) or of a
tile, groups across two tiles, every number of Gauss points, stencils
shorter than the ring of requests, cells with 3 to 16 face slots; and the
two storage orders of the coefficients, which must hold the same values.

Bars: the residual within 1e-12 of the largest force sum, as everywhere
(products to 2^-48, sums to a few 2^-48 of their terms); a pair holds its
FP64 value to 2^-48."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2601_18417_gb300 import hofv
from paper_2601_18417_gb300 import inputs as I
from tests import helpers as H
from tests.test_gpu_parity import smooth_u

pytestmark = pytest.mark.gpu

# dim, cells, n, p, n_plus, q, law
CASES = {
    "quad-q1-short": (2, "tensor", 5, 1, 2, 1, 0),
    "quad-q2": (2, "tensor", 7, 2, 10, 2, 1),
    "quad-q3-long": (2, "tensor", 9, 3, 30, 3, 0),
    "quad-q4": (2, "tensor", 6, 2, 9, 4, 0),
    "tri-q3": (2, "simplex", 5, 3, 10, 3, 0),
    "poly-q2": (2, "polygon", 7, 2, 10, 2, 0),
    "hex-q1-short": (3, "tensor", 3, 1, 2, 1, 1),
    "hex-q2": (3, "tensor", 5, 2, 31, 2, 1),
    "hex-q3": (3, "tensor", 5, 2, 40, 3, 0),
    "tet-q2": (3, "simplex", 3, 2, 40, 2, 0),
    "hexfaces-q1": (3, "hexfaces", 4, 1, 20, 1, 0),
    "hexfaces-q2": (3, "hexfaces", 4, 2, 30, 2, 1),
    "prism-q1": (3, "polyhedron", 4, 1, 20, 1, 1),
    "prism-q2": (3, "polyhedron", 4, 2, 40, 2, 0),
}


def _make(name):
    dim, kind, n, p, n_plus, q, law = CASES[name]
    tags = I.side_tags("block" if law == 1 else "mms", dim)
    mu, lam = (1e6, 4e6) if law == 1 else (1.0, 1.5)
    pb = H.make_problem(dim, n, p, q, n_plus=n_plus, jitter=0.1, seed=3, field=None, tags=tags,
                        law=law, mu=mu, lam=lam, kind=kind)
    rng = np.random.default_rng(8)
    pb.ubq = 1e-2 * rng.standard_normal(pb.ubq.shape)
    pb.ubf = 1e-2 * rng.standard_normal(pb.ubf.shape)
    return pb, H.gpu_context(pb)


def _residual(ctx, u):
    import torch
    ud = H.to_dev(u)
    R = torch.full_like(ud, float("nan"))
    ctx.residual(ud, R)
    return R.cpu().numpy()


@pytest.mark.parametrize("name", list(CASES))
def test_residual_at_group_edges(name):
    pb, ctx = _make(name)
    ctx.set_precision(hofv.PREC_DF64)
    u = smooth_u(pb, 1, amp=1e-2)
    ref = H.residual(pb, u)
    Fs = H.force_scale(pb.orc, pb.law, pb.mu, pb.lam, u, pb.ubq, pb.ubf, pb.tbq)
    assert np.abs(_residual(ctx, u) - ref).max() <= 1e-12 * Fs


@pytest.mark.parametrize("name", ["quad-q3-long", "tri-q3", "poly-q2", "hex-q2", "tet-q2", "prism-q2"])
def test_storage_orders_hold_the_same_coefficients(name):
    pb, ctx = _make(name)
    lay = ctx.layout
    nf = lay.n_internal + lay.n_disp
    _, co = ctx.get_face_data(0, nf)
    _, ex = ctx.get_cell_data(0, lay.n_cells)
    u = smooth_u(pb, 2, amp=1e-2)
    ctx.set_precision(hofv.PREC_DF64)
    _, co_df = ctx.get_face_data(0, nf)
    _, ex_df = ctx.get_cell_data(0, lay.n_cells)
    S = lay.stencil
    assert np.all(np.abs(co_df[:, :, :S] - co[:, :, :S]) <= 2.0 ** -48 * np.abs(co[:, :, :S]))
    assert np.all(np.abs(ex_df - ex) <= 2.0 ** -48 * np.abs(ex))
    R_df = _residual(ctx, u)
    ctx.set_precision(hofv.PREC_FP64)  # the pairs' values, as doubles in their own order
    assert np.array_equal(ctx.get_face_data(0, nf)[1], co_df)
    assert np.array_equal(ctx.get_cell_data(0, lay.n_cells)[1], ex_df)
    ctx.set_precision(hofv.PREC_DF64)
    assert np.array_equal(_residual(ctx, u), R_df)


@pytest.mark.parametrize("name", ["quad-q2", "hex-q2"])
def test_new_stencils_in_double_float_order(name):
    """The fits write doubles over the pairs' order; the residual is the same
    as before when the stencils are."""
    pb, ctx = _make(name)
    lay = ctx.layout
    ctx.set_precision(hofv.PREC_DF64)
    u = smooth_u(pb, 2, amp=1e-2)
    R = _residual(ctx, u)
    st, _ = ctx.get_face_data(0, lay.n_internal + lay.n_disp, coef=False)
    cst, _ = ctx.get_cell_data(0, lay.n_cells, ext=False)
    ctx.set_stencils(st, cst)
    assert np.array_equal(_residual(ctx, u), R)
