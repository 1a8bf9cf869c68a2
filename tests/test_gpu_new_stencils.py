"""Stencils replaced while the coefficients lie in the double-float order, on
cells whose face slots are partly empty: the weights of a slot without a face
are zero (hofv_get_cell_data), before and after, and the same stencils give
the same coefficients bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2601_18417_gb300 import hofv
from tests.test_gpu_face_groups import _make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["poly-q2", "hexfaces-q2", "prism-q2", "quad-q2"])
def test_the_same_stencils_give_the_same_coefficients(name):
    pb, ctx = _make(name)
    lay = ctx.layout
    nf = lay.n_internal + lay.n_disp
    sides = (pb.orc.cell_faces() >= 0).sum(axis=1)
    empty = np.arange(ctx.faces_per_cell)[None, :] >= sides[:, None]
    assert empty.any() == (name != "quad-q2")
    ctx.set_precision(hofv.PREC_DF64)
    st, co = ctx.get_face_data(0, nf)
    cst, ex = ctx.get_cell_data(0, lay.n_cells)
    assert not ex[empty].any()
    for faces, cells in ((st, cst), (None, cst), (st, None)):
        ctx.set_stencils(faces, cells)
        assert np.array_equal(ctx.get_face_data(0, nf)[1], co)
        assert np.array_equal(ctx.get_cell_data(0, lay.n_cells)[1], ex)
    ctx.set_precision(hofv.PREC_FP64)
    assert np.array_equal(ctx.get_cell_data(0, lay.n_cells)[1], ex)
    ctx.close()
