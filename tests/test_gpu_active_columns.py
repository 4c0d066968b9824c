"""A preconditioner whose active columns change under a solver or a batch that
has captured its launches: later steps use the new columns, whichever way the
count went, with the scratch that was reserved at creation."""
import numpy as np
import pytest

from gpu_util import require_gpu
from workloads import gaussian_kernel, phantom

pytestmark = pytest.mark.gpu

# below 1/4, so that sqrt(s_last) exceeds every s_i: no column is active with
# the square-rooted shift, all but the last without
EIGS = (0.24, 0.1)


def factor(torch, api, ctx, N, ell, dtype, shift):
    U = np.linalg.qr(np.random.default_rng(N + ell).standard_normal((N, ell)))[0].T
    pc = api.Precond(ctx, N, ell, dtype).import_factor(U, np.geomspace(*EIGS, ell), 0.0, shift)
    assert pc.ell_active == (0 if shift else ell - 1)
    return pc


@pytest.mark.parametrize("grow", [True, False])
@pytest.mark.parametrize("reg,n,ell,dt", [("wavelet", 64, 32, "float64"), ("wavelet", 64, 128, "float32"),
                                          ("wavelet", 256, 40, "float32"), ("tv", 64, 32, "float32"),
                                          ("tv", 64, 100, "float32"), ("hs", 33, 20, "float64"),
                                          ("tv", 33, 20, "float32")])
def test_solver(reg, n, ell, dt, grow):
    torch, api = require_gpu()
    dtype = getattr(torch, dt)
    ctx, ref_ctx = api.Context(0), api.Context(0)
    kw = dict(alpha=0.4, n_inner=5)

    def make(c, pc):
        op = api.Operator(c, "blur", n, n, dtype=dtype, kernel=gaussian_kernel(7, 1.5),
                          haar_levels=3 if reg == "wavelet" else 0)
        y = torch.from_numpy(phantom(n, 5, 1, "mixed")).to(dtype).cuda()
        return api.Solver(c, op, y, reg, 1e-2, pc=pc, **kw)

    pc = factor(torch, api, ctx, n * n, ell, dtype, grow)
    sol = make(ctx, pc)
    sol.step(2)
    pc.setup(0.0, not grow)
    sol.restart()
    sol.step(3)
    ref = make(ref_ctx, factor(torch, api, ref_ctx, n * n, ell, dtype, not grow))
    ref.step(3)
    assert torch.equal(sol.x(), ref.x())


@pytest.mark.parametrize("grow", [True, False])
@pytest.mark.parametrize("n,ell", [(64, 12), (64, 100), (33, 20)])
def test_batch(n, ell, grow):
    torch, api = require_gpu()
    main = api.Context(0, torch.cuda.Stream(priority=-1))
    stream = torch.cuda.Stream()
    ctx = api.Context(0, stream)
    with torch.cuda.stream(stream):
        op = api.Operator(ctx, "blur", n, n, dtype=torch.float32, kernel=gaussian_kernel(7, 1.5))
        pc = factor(torch, api, ctx, n * n, ell, torch.bfloat16, grow)
        un = api.Unroll(ctx, op, 1e-2, 0.4, 3, n_inner=3, ckpt_every=2, pc=pc)
        y = torch.from_numpy(phantom(n, 5, 1, "mixed")).float().cuda()
        x, xbar = torch.zeros_like(y), torch.ones_like(y)
    torch.cuda.synchronize()
    B = api.Batch(main, [un], [y], [x], [xbar])
    B.forward()
    B.backward()
    torch.cuda.synchronize()
    first = x.clone()
    with torch.cuda.stream(stream):
        pc.setup(0.0, not grow)
    torch.cuda.synchronize()
    B.forward()
    B.backward()
    torch.cuda.synchronize()
    got, g = x.clone(), B.grads[0].clone()
    with torch.cuda.stream(stream):
        ref = un.forward(y)
        dl, dh = un.backward(xbar)
    torch.cuda.synchronize()
    assert torch.equal(got, ref) and not torch.equal(got, first)
    assert float(g[0]) == float(dl) and torch.equal(g[1:], dh.reshape(-1))
