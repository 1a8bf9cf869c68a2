"""The vector kernels of a flexible Arnoldi step at basis sizes on both sides of
the four vectors a block of the multi-dot takes, on meshes below and above one
pass of its blocks: the step's column against the product and FP64 dots, and the
orthogonality of the next vector."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

from paper_2601_18417_gb300 import hofv  # noqa: E402
from tests import helpers as H  # noqa: E402


@pytest.mark.parametrize("prec", [hofv.PREC_FP64, hofv.PREC_DF64])
@pytest.mark.parametrize("dim,n,p,q1", [(2, 5, 2, 2), (2, 151, 2, 2), (3, 7, 2, 2)])
def test_step_against_dots(dim, n, p, q1, prec):
    pb = H.make_problem(dim, n, p, q1, jitter=0.1, seed=4)
    ctx = H.gpu_context(pb)
    ctx.set_precision(prec)
    rng = np.random.default_rng(8)
    N = pb.u_exact.size
    u = H.to_dev(rng.standard_normal(pb.u_exact.shape))
    R, Jv = torch.empty_like(u), torch.empty_like(u)
    ctx.residual(u, R)
    kmax = 10
    V0 = torch.linalg.qr(H.to_dev(rng.standard_normal((N, kmax + 1))))[0].T.contiguous()
    for k in (1, 2, 3, 4, 5, 8, 9):
        V = V0[: k + 1].clone()
        Z = torch.zeros_like(V)
        h = np.asarray(ctx.arnoldi_step(u, R, hofv.PC_NONE, 0, V, Z, k - 1))
        assert torch.equal(Z[k - 1], V[k - 1])
        ctx.jvp(u, R, Z[k - 1].reshape(u.shape), Jv)
        w = Jv.reshape(-1).cpu().numpy()
        B, v = V[:k].cpu().numpy(), V[k].cpu().numpy()
        # dots of N terms and two projections in FP64: N 2^-52 at most, of |w|
        tol = N * 2.0 ** -52 * np.linalg.norm(w)
        assert np.abs(B @ w - h[:k]).max() <= tol
        assert abs(np.linalg.norm(v) - 1.0) <= N * 2.0 ** -52
        assert np.abs(B @ v).max() * h[k] <= tol
        assert np.linalg.norm(w - B.T @ h[:k] - h[k] * v) <= np.sqrt(N) * tol
    ctx.close()
