"""The wavelet prox's Newton iteration at the ends of its two paths (one cluster
launch while the active columns fit its shared memory, evaluation and step
launches beyond), with few, all and no active columns, ragged pixel slices,
thresholds from weak to saturating and starts away from zero, against the
float64 oracle."""
import numpy as np
import pytest

import oracle.nystrom
import oracle.prox
from gpu_util import rel, require_gpu

pytestmark = pytest.mark.gpu

# (N, ell, sqrt_shift, largest / smallest eigenvalue): slices of one pixel to
# 4096 pixels a CTA, 1 to 128 columns, factors either side of 220 KB a CTA
CASES = [
    (16, 1, True, 4.0),
    (17, 5, False, 30.0),
    (1000, 33, False, 50.0),
    (4096, 32, True, 900.0),
    (4099, 64, False, 20.0),
    (4096, 128, False, 40.0),
    (2048, 127, True, 1e4),
    (65536, 6, True, 1e3),
    (65536, 40, False, 1e3),
    (512, 9, True, 1.0),
]


@pytest.fixture(scope="module")
def env():
    torch, api = require_gpu()
    return torch, api, api.Context(0)


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("N,ell,shift,ratio", CASES)
@pytest.mark.parametrize("tau", [1e-3, 0.3])
def test_prox_wavelet(env, N, ell, shift, ratio, tau, dt):
    torch, api, ctx = env
    rng = np.random.default_rng(N + ell)
    U = np.linalg.qr(rng.standard_normal((N, ell)))[0].T
    S = np.geomspace(ratio, 1.0, ell) if ratio > 1.0 else np.full(ell, 0.25)   # 0.25: sqrt(s) above every s
    s = rng.standard_normal(N)
    tdt = torch.float64 if dt == "f64" else torch.float32
    if dt == "f32":
        U, s = U.astype(np.float32).astype(np.float64), s.astype(np.float32).astype(np.float64)
    pc = api.Precond(ctx, N, ell, tdt).import_factor(U, S, 0.0, shift)
    P = oracle.nystrom.Precond(U, S, 0.0, shift)
    x_ref, g_ref, _, ok = oracle.prox.prox_wavelet(s, P.Ubar, tau)
    assert ok
    g0 = torch.from_numpy(rng.standard_normal(ell)).cuda()
    x, info = api.prox_wavelet(ctx, pc, tau, torch.from_numpy(s).to(tdt).cuda(), gamma=g0)
    assert info["converged"]
    # the Newton tolerance (1e-12 or 1e-6 of 1 + ||Ubar^T s||) carried to x
    scale = 1.0 + np.linalg.norm(P.Ubar @ s)
    tol = (1e-12 if dt == "f64" else 1e-6) * scale * max(1.0, np.sqrt(P.d.max())) / np.linalg.norm(x_ref) + \
        (1e-13 if dt == "f64" else 1e-6)
    assert rel(x.cpu(), x_ref) < 10.0 * tol
    assert np.linalg.norm(g0.cpu().numpy() - g_ref) <= 10.0 * (1e-12 if dt == "f64" else 1e-6) * scale
