"""The ell x ell part of Algorithm 1 at the edges of its blocks (panels of 32,
product tiles of 16, inverses of 128, 256 and 512) against numpy in float64: C
and its inverse through W = C^{-T} V S^{-1} from a Gram with a known factor, and
the retries when the first shift is too small."""
import numpy as np
import pytest

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch, api = require_gpu()
    return torch, api, api.Context(0)


def gram(ell, seed, N=None):
    rng = np.random.default_rng(seed)
    N = N or 4 * ell + 40
    Om = rng.standard_normal((ell, N))
    Y = Om * np.geomspace(1.0, 1e-2, N)          # Phi diagonal, positive
    A = np.concatenate([Om, Y])
    return A @ A.T, Om, Y


@pytest.mark.parametrize("ell", [1, 2, 15, 16, 17, 31, 32, 33, 48, 64, 65, 127, 128, 129, 200, 256, 257, 400, 513])
@pytest.mark.parametrize("f64", [True, False])
def test_factor_from_gram(env, ell, f64):
    torch, api, ctx = env
    if f64 and ell > 257:
        pytest.skip("the float64 eigensolver takes seconds here")
    G2, Om, Y = gram(ell, ell)
    eps = 2.0 ** -30
    W, S, v, retries = api.nys_factor_gram(ctx, torch.from_numpy(G2).cuda(), ell, eps, eig_f64=f64)
    W, S = W.cpu().numpy(), S.cpu().numpy()
    v_ref = eps * np.linalg.norm(Om)
    assert retries == 0 and abs(v - v_ref) <= 1e-12 * v_ref
    Yv = Y + v * Om
    M = Om @ Yv.T
    C = np.linalg.cholesky(0.5 * (M + M.T))
    B = np.linalg.solve(C, Yv)
    s2 = np.sort(np.linalg.eigvalsh(B @ B.T))[::-1]
    if f64:
        assert np.max(np.abs(S - np.maximum(s2 - v, 0.0))) <= 1e-11 * s2[0]
    # the eigenvalues are the float64 Rayleigh quotients of the vectors returned,
    # V = C^T W diag(S): sums of ell^2 products in float64
    V = C.T @ W
    lam = np.einsum("ri,rs,si->i", V, B @ B.T, V) / np.einsum("ri,ri->i", V, V)
    assert np.max(np.abs(S - np.maximum(lam - v, 0.0))) <= 1e-11 * s2[0]
    if f64:
        # U = Yv^T W: orthonormal columns that reproduce Yv (Om^T Yv)^{-1} Yv^T
        U = W.T @ Yv
        assert np.max(np.abs(U @ U.T - np.eye(ell))) <= 1e-10
        z = np.random.default_rng(1).standard_normal(Om.shape[1])
        ref = B.T @ (B @ z)
        got = U.T @ ((S + v) * (U @ z))
        assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("ell", [20, 100, 520])
def test_retries(env, ell):
    torch, api, ctx = env
    G2, Om, Y = gram(ell, 7)
    # push the core's smallest eigenvalue below -v for the first two shifts
    n = ell
    M = 0.5 * (G2[:n, n:] + G2[n:, :n])
    eps = 1e-6
    v0 = eps * np.sqrt(np.trace(G2[:n, :n]))
    lam = np.linalg.eigvals(np.linalg.solve(G2[:n, :n], M)).real.min()
    G2[:n, n:] -= (lam + 30.0 * v0) * G2[:n, :n]
    G2[n:, :n] = G2[:n, n:].T
    _, _, v, retries = api.nys_factor_gram(ctx, torch.from_numpy(G2).cuda(), ell, eps)
    assert retries == 2 and abs(v - 100.0 * v0) <= 1e-9 * v0
