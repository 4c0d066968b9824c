"""What a ray operator allocates is bounded by a few images where the images are
large, and batches that its scratch then cuts into smaller chunks give the
images' own results."""
import math

import numpy as np
import pytest

from gpu_util import TOL, require_gpu

pytestmark = pytest.mark.gpu


def make(torch, api, kind, n1, n2, dt, A, B, span=None):
    kw = {}
    if kind == "fanbeam":
        r = math.hypot(n1, n2)
        kw = dict(src_dist=r, det_dist=2.0 * r, det_spacing=2.2 * r / B)
    return api.Operator(api.Context(0), kind, n1, n2, dtype=getattr(torch, dt), n_angles=A, n_bins=B, angle_span=span, **kw)


@pytest.mark.parametrize("kind,n,dt,images", [("fanbeam", 4096, "float64", 21), ("radon", 4096, "float64", 21),
                                              ("radon", 6144, "float32", 21), ("fanbeam", 512, "float32", 90)])
def test_bytes_at_creation(kind, n, dt, images):
    """Twenty images (two copies of eight lanes, four planes) and one more for margins
    and tables; 32 images' lines where they are small."""
    torch, api = require_gpu()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    make(torch, api, kind, 64, 64, dt, 8, 128)          # the kernels' module and the context
    free = torch.cuda.mem_get_info()[0]
    op = make(torch, api, kind, n, n, dt, 8, 128)
    used = free - torch.cuda.mem_get_info()[0]
    assert used <= images * n * n * (8 if dt == "float64" else 4) + (64 << 20)
    op.close()


@pytest.mark.parametrize("kind,n1,n2,span,batch", [("radon", 2080, 2080, None, 31), ("radon", 2200, 1990, None, 31),
                                                   ("radon", 2080, 2080, 2.0, 30), ("fanbeam", 2080, 2080, None, 31)])
def test_chunked_batch(kind, n1, n2, span, batch):
    """More images than a chunk and a rest of two or three, each against itself: two
    float64 results, each held to 1e-12, differ by twice that at most."""
    torch, api = require_gpu()
    op = make(torch, api, kind, n1, n2, "float64", 6, 96, span)
    g = torch.Generator(device="cuda").manual_seed(n1)
    x = torch.randn((batch, n1, n2), dtype=torch.float64, device="cuda", generator=g)
    s = torch.randn((batch, 6, 96), dtype=torch.float64, device="cuda", generator=g)
    y, z = api.op_apply(op, x), api.op_adjoint(op, s)
    for b in (0, 7, 27, 28, batch - 2, batch - 1):
        for got, one in ((y[b], api.op_apply(op, x[b:b + 1])[0]), (z[b], api.op_adjoint(op, s[b:b + 1])[0])):
            assert float((got - one).abs().max()) <= 2.0 * TOL["f64"] * float(one.abs().max())
    assert np.isfinite(float(y.sum()))
