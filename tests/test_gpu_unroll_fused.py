"""The fused passes of the unrolled solve where they can go wrong: sides of one,
two and odd lengths (the periodic neighbours of an edge, a pixel that is its own
neighbour), 0, 1, 2 and 3 dual steps (the ping-pong's ends), with and without a
preconditioner, sizes its vectorised apply takes and refuses, against the
float64 oracle's forward and hand-derived gradient."""
import numpy as np
import pytest

import oracle
import oracle.nystrom
import oracle.operators as O
import oracle.unroll
from gpu_util import rel, require_gpu
from workloads import random_kernel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch, api = require_gpu()
    return torch, api, api.Context(0)


@pytest.mark.parametrize("n1,n2,ell", [(1, 3, 0), (2, 2, 2), (5, 7, 0), (16, 12, 5), (9, 9, 4), (33, 20, 70), (64, 65, 0)])
@pytest.mark.parametrize("J", [0, 1, 2, 3])
def test_forward_and_gradient(env, n1, n2, ell, J):
    torch, api, ctx = env
    rng = np.random.default_rng(n1 * 100 + n2 + J)
    h = random_kernel(1 if min(n1, n2) < 3 else 3, 4)
    opo = O.Operator("blur", n1, n2, kernel=h)
    op = api.Operator(ctx, "blur", n1, n2, dtype=torch.float64, kernel=h)
    y = rng.uniform(size=(n1, n2))
    x_ref = rng.uniform(size=(n1, n2))
    pc, P = None, oracle.nystrom.Identity()
    if ell:
        U = np.linalg.qr(rng.standard_normal((n1 * n2, ell)))[0].T
        S = np.geomspace(3.0, 1.0, ell)
        pc = api.Precond(ctx, n1 * n2, ell, torch.float64).import_factor(U, S, 0.0, False)
        P = oracle.nystrom.Precond(U, S, 0.0, False)
    K, lam, alpha = 4, 0.05, 0.3
    un = api.Unroll(ctx, op, lam, alpha, K, n_inner=J, ckpt_every=3, pc=pc)
    x = un.forward(torch.from_numpy(y).cuda())
    xr, _ = oracle.unroll.forward(opo, y, lam, alpha, P, K, J)
    assert rel(x, xr) < 1e-12
    _, rl, rh = oracle.unroll.value_and_grad(opo, y, lam, alpha, P, K, J, x_ref)
    gl, gh = un.backward(torch.from_numpy(2.0 * (xr - x_ref) / (n1 * n2)).cuda())
    assert abs(float(gl) - rl) <= 1e-9 * max(1.0, abs(rl))
    assert rel(gh, rh) < 1e-9
