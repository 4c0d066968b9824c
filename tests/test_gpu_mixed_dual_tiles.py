"""The one-launch dual step of the mixed norms without a preconditioner at the
edges of its 32 x 16 tiles: sides of one pixel (every neighbour is the pixel
itself) to a little over two tiles, 0 to 5 steps, warm starts, against the
float64 oracle, and with the exact early stop on and off bit for bit."""
import numpy as np
import pytest

import oracle.nystrom
import oracle.prox
from gpu_util import rel, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch, api = require_gpu()
    return torch, api, api.Context(0)


@pytest.mark.parametrize("reg", ["isotv", "hs", "hs2", "hsinf"])
@pytest.mark.parametrize("n1,n2", [(1, 1), (1, 5), (2, 2), (3, 33), (16, 32), (17, 31), (33, 65), (40, 70)])
@pytest.mark.parametrize("steps,lam", [(0, 0.1), (1, 0.1), (2, 0.5), (5, 0.05), (40, 1e-6)])
def test_prox(env, reg, n1, n2, steps, lam):
    torch, api, ctx = env
    G = 2 if reg == "isotv" else 3
    rng = np.random.default_rng(n1 * 100 + n2)
    s = rng.standard_normal((n1, n2))
    Q0 = 0.3 * rng.standard_normal((G, n1, n2))
    x_ref, Q_ref = oracle.prox.prox_dual(s, reg, lam, oracle.nystrom.Identity(), steps, Q0)
    got = []
    for stop in (True, False):
        ctx.set_dual_stop(stop)
        Q = torch.from_numpy(Q0).cuda()
        x, Q = api.prox_mixed(ctx, None, reg, lam, steps, torch.from_numpy(s).cuda(), Q=Q)
        got.append((x.clone(), Q.clone()))
    ctx.set_dual_stop(True)
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    x, Q = got[0]
    # lam / step scale: errors in z are those of x over 8 lam (32 lam)
    assert rel(x, x_ref) < 1e-12
    assert np.max(np.abs(Q.cpu().numpy() - Q_ref)) < 1e-15 / lam * 10.0 * np.abs(s).max() + 1e-12
