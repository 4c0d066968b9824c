"""The blur kernels at the edges of their tile and strip choices: sides around
64 and 128, kernels from 1 to 33 taps (remainders of every residue modulo 8 in
the normal operator), odd batches, separable and general, against the float64
oracle; and the strips against the tiles bit for bit (the same sums in the same
order)."""
import numpy as np
import pytest

import oracle.operators as O
from gpu_util import TOL, close, require_gpu
from workloads import gaussian_kernel, random_kernel

pytestmark = pytest.mark.gpu

# (n1, n2, kh, kw, batch): small work (tiles of 8 .. 64), then enough images for strips
CASES = [
    (8, 8, 3, 3, 1), (64, 64, 9, 9, 1), (65, 40, 5, 7, 3), (130, 257, 13, 25, 1),
    (64, 65, 1, 9, 400), (65, 128, 5, 3, 300), (100, 129, 7, 11, 200), (127, 191, 15, 13, 110), (192, 64, 33, 33, 230),
    (200, 300, 25, 17, 40), (70, 72, 31, 29, 320),
]


@pytest.fixture(scope="module")
def env():
    torch, api = require_gpu()
    return torch, api, api.Context(0)


def kernel(kh, kw, separable):
    if not separable:
        return random_kernel(max(kh, kw), 5)[:kh, :kw]
    # exactly rank one in float64: weights that are multiples of a power of two
    u = np.round(gaussian_kernel(kh, kh / 5)[kh // 2] * 4096) + 1.0
    v = np.round(gaussian_kernel(kw, kw / 5)[kw // 2] * 4096) + 2.0
    v[0] += 1.0                      # not symmetric: H and H^T differ
    return np.outer(u / u.sum(), v / v.sum())


@pytest.mark.parametrize("dt", ["f32", "f64"])
@pytest.mark.parametrize("separable", [True, False])
@pytest.mark.parametrize("case", CASES)
def test_blur(env, case, separable, dt):
    torch, api, ctx = env
    n1, n2, kh, kw, batch = case
    if batch > 3 and (dt == "f64" or not separable):
        batch = 2
    h = kernel(kh, kw, separable)
    op = api.Operator(ctx, "blur", n1, n2, dtype=getattr(torch, {"f32": "float32", "f64": "float64"}[dt]), kernel=h)
    x = np.random.default_rng(n1 + kh).standard_normal((batch, n1, n2))
    xt = torch.from_numpy(x).to(op.dtype).cuda()
    pick = [0, batch - 1]
    hx = O.blur_apply(x[pick], h)
    close(api.op_apply(op, xt)[pick], hx, TOL[dt])
    close(api.op_adjoint(op, xt)[pick], O.blur_adjoint(x[pick], h), TOL[dt])
    full = api.op_normal(op, xt)
    close(full[pick], O.blur_adjoint(hx, h), TOL[dt])
    # one image at a time takes tiles
    for b in pick:
        assert torch.equal(api.op_normal(op, xt[b:b + 1].contiguous())[0], full[b])
