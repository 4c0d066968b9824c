"""Pivots of the preconditioner's Cholesky over float64's range: a weight near the
largest finite number (its pivot's reciprocal is subnormal) and ordinary ones
beside it, against P^{-1} z = z - sum_i d_i / (1 + d_i) u_i (u_i^T z) for
orthonormal u_i."""
import numpy as np
import pytest

from gpu_util import TOL, rel, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top", [1e3, 1e150, 1e307, 8e307, 1.7e308])
@pytest.mark.parametrize("ell", [3, 33, 70])
def test_setup(top, ell):
    torch, api = require_gpu()
    ctx = api.Context(0)
    N = 256
    rng = np.random.default_rng(ell)
    U = np.linalg.qr(rng.standard_normal((N, ell)))[0].T
    S = np.concatenate([[top], np.linspace(9.0, 1.0, ell - 1)])
    pc = api.Precond(ctx, N, ell, torch.float64).import_factor(U, S, 0.0, False)
    z = rng.standard_normal((2, N))
    d = S / S[-1] - 1.0
    ref = z - ((z @ U.T) * (d / (1.0 + d))) @ U
    out = api.precond_apply(ctx, pc, torch.from_numpy(z).cuda())
    assert rel(out.cpu().numpy(), ref) <= TOL["f64"]
