"""A NaN, an infinite or a very large value of one cell in double-float mode
reaches the cells that see it through a stencil and no other, whatever the
cell's number: those cells are the ones the default precision loses too, and
all others keep their residual and product bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2601_18417_gb300 import hofv
from tests import helpers as H
from tests.test_gpu_face_groups import CASES, _make, _residual
from tests.test_gpu_parity import smooth_u

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["quad-q3-long", "tri-q3", "poly-q2", "hex-q2", "tet-q2", "prism-q2"])
def test_bad_values_stay_local(name):
    import torch
    pb, ctx = _make(name)
    u = smooth_u(pb, 1, amp=1e-2)
    v = np.random.default_rng(3).standard_normal(u.shape)
    linear = CASES[name][-1] == 0

    def product(w):
        R, out = torch.empty_like(H.to_dev(u)), torch.full_like(H.to_dev(u), float("nan"))
        ud = H.to_dev(u)
        ctx.residual(ud, R)
        ctx.jvp(ud, R, H.to_dev(w), out)
        return out.cpu().numpy()

    for cell in (0, u.shape[1] // 2, u.shape[1] - 1):
        bad = u.copy()
        bad[1, cell] = np.nan
        ctx.set_precision(hofv.PREC_FP64)
        hit = ~np.isfinite(_residual(ctx, bad)).all(axis=0)
        assert hit[cell]
        ctx.set_precision(hofv.PREC_DF64)
        base, base_v = _residual(ctx, u), product(v) if linear else None
        for value in (np.nan, np.inf, -np.inf, 1e300):
            bad[1, cell] = value
            r = _residual(ctx, bad)
            if not np.isfinite(value):
                assert np.array_equal(~np.isfinite(r).all(axis=0), hit)
            assert np.array_equal(r[:, ~hit], base[:, ~hit])
            if linear:  # the homogeneous residual of v: no norm of v in it
                w = v.copy()
                w[1, cell] = value
                assert np.array_equal(product(w)[:, ~hit], base_v[:, ~hit])
    ctx.close()
