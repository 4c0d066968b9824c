"""Blur + decimation where the taps wrap: images smaller than the kernel (more
than once around), kernels whose taps are no multiple of the groups that load
together, and phases with no tap at all, against the float64 oracle."""
import numpy as np
import pytest

import oracle.operators as O
from gpu_util import TOL, close, require_gpu
from workloads import random_kernel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["f32", "f64"])
@pytest.mark.parametrize("n1,n2,kh,kw,d,batch", [
    (4, 4, 9, 11, 4, 1), (2, 6, 7, 1, 2, 3), (3, 3, 1, 1, 3, 2), (12, 8, 3, 25, 4, 1), (30, 45, 17, 9, 15, 2),
    (64, 96, 7, 7, 1, 2), (128, 132, 23, 15, 4, 5),
])
def test_apply_adjoint_normal(dt, n1, n2, kh, kw, d, batch):
    torch, api = require_gpu()
    ctx = api.Context(0)
    h = random_kernel(max(kh, kw), 7)[:kh, :kw]
    rng = np.random.default_rng(n1 + kh)
    x, y = rng.standard_normal((batch, n1, n2)), rng.standard_normal((batch, n1 // d, n2 // d))
    dtype = torch.float64 if dt == "f64" else torch.float32
    op = api.Operator(ctx, "blur_decim", n1, n2, dtype=dtype, kernel=h, decim=d)
    xt, yt = (torch.from_numpy(v).to(dtype).cuda() for v in (x, y))
    got = [api.op_apply(op, xt), api.op_adjoint(op, yt), api.op_normal(op, xt)]
    fwd = [O.decim_apply(v, h, d) for v in x]
    want = [fwd, [O.decim_adjoint(v, h, d) for v in y], [O.decim_adjoint(v, h, d) for v in fwd]]
    for g, w in zip(got, want):
        close(g.cpu().reshape(np.shape(w)), np.stack(w), TOL[dt])
