"""The fixed-point contractions of the default precision (HOFV_PREC_FP64): the
residual of the linear law against the oracle for states whose values differ
widely in size, exact scaling with powers of two inside the range of the
fixed-point scales, and the FP64 sums outside it (tiny, huge, infinite and NaN
values, all-zero components)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

from tests import helpers as H  # noqa: E402


def _residual(ctx, u):
    ud = H.to_dev(u)
    R = torch.empty_like(ud)
    ctx.residual(ud, R)
    torch.cuda.synchronize()
    return R.cpu().numpy()


def _problem(dim, n, p, q1, jitter=0.2):
    """A block without data: zero prescribed displacements, no body force."""
    pb = H.make_problem(dim, n, p, q1, jitter=jitter, seed=3)
    return pb, H.gpu_context(pb)


SCHEMES = [(2, 9, 1, 1), (2, 33, 2, 2), (2, 17, 3, 3), (2, 12, 3, 4), (3, 5, 1, 1), (3, 7, 2, 2), (3, 6, 3, 3)]


@pytest.mark.parametrize("dim,n,p,q1", SCHEMES)
@pytest.mark.parametrize("spread", [0, 40])
def test_against_oracle(dim, n, p, q1, spread):
    """A slot's error is at most 2^-53 of its face's largest coefficient times
    its largest value, below the bound of an FP64 sum: the tolerance is the
    1e-12 of the force scale that FP64 residuals are held to elsewhere."""
    pb, ctx = _problem(dim, n, p, q1)
    g = np.random.default_rng(5)
    u = g.standard_normal(pb.u_exact.shape) * 2.0 ** -g.integers(0, spread + 1, pb.u_exact.shape)
    ref = H.residual(pb, u)
    Fs = H.force_scale(pb.orc, 0, 1.0, 1.5, u, pb.ubq, pb.ubf, pb.tbq)
    assert np.abs(_residual(ctx, u) - ref).max() <= 1e-12 * Fs
    ctx.close()


@pytest.mark.parametrize("dim,n,p,q1", SCHEMES)
def test_scaling_zero_and_non_finite(dim, n, p, q1):
    pb, ctx = _problem(dim, n, p, q1)
    nc = pb.u_exact.shape[1]
    g = np.random.default_rng(6)
    u = g.standard_normal(pb.u_exact.shape)
    u[0] = 0.0                                   # a component without any value
    assert not _residual(ctx, np.zeros_like(u)).any()
    base = _residual(ctx, u)
    assert np.isfinite(base).all()
    for k in (300, -300):                        # fixed point: every rounding scales along
        assert np.array_equal(_residual(ctx, u * 2.0 ** k), base * 2.0 ** k)
    Fs = H.force_scale(pb.orc, 0, 1.0, 1.5, u, pb.ubq, pb.ubf, pb.tbq)
    for k in (600, -600, -990):                  # FMAs
        assert np.abs(_residual(ctx, u * 2.0 ** k) - base * 2.0 ** k).max() <= 1e-12 * Fs * 2.0 ** k
    # cells that see an infinite or NaN value lose their finite residual, the
    # others keep theirs bit for bit
    for bad in (np.nan, np.inf, -np.inf):
        v = u.copy()
        v[1, nc // 2] = bad
        r = _residual(ctx, v)
        hit = ~np.isfinite(r).all(axis=0)
        assert hit[nc // 2]
        assert np.array_equal(r[:, ~hit], base[:, ~hit])
    ctx.close()
