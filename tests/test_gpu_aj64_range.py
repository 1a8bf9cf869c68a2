"""The FP64 approximate-Jacobian solve at the ends of the range of its inner
products (gamma = r^T D^-1 r): right-hand sides so small that gamma is a
subnormal number, and far more iterations than the recurrence needs to
converge, on a mesh of one block and one of several."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2601_18417_gb300 import hofv
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(2, 8), (3, 12)])
def test_tiny_right_hand_side_and_many_iterations(dim, n):
    import torch
    pb = H.make_problem(dim, n, 1, 1, jitter=0.1, seed=2, prepare=False)
    ctx = H.gpu_context(pb)
    v = H.to_dev(np.random.default_rng(4).standard_normal((dim, pb.orc.nc)))
    z, ref = torch.empty_like(v), torch.empty_like(v)
    ctx.precondition(hofv.PC_AJ64, 4, v, ref)
    for k in (1e-154, 1e-155, 1e-156):
        ctx.precondition(hofv.PC_AJ64, 4, v * k, z)
        # a subnormal gamma of 1e-313 has 2e-11 of its value as spacing
        assert ((z / k - ref).norm() <= 1e-6 * ref.norm()).item(), k
    for iters in (300, 1000):
        ctx.precondition(hofv.PC_AJ64, iters, v, z)
        assert torch.isfinite(z).all().item(), iters
    ctx.close()
