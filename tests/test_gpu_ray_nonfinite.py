"""An infinity or a NaN in one bin of a sinogram reaches the pixels that its ray
touches and no others (both ray transforms, single images in mirror lanes and
batches)."""
import math

import numpy as np
import pytest

import oracle.operators as O
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

GEOMS = [("radon", 48, 48, 12, 70, {}), ("radon", 40, 33, 7, 64, {}), ("radon", 64, 64, 9, 97, {"angle_span": 2.0}),
         ("fanbeam", 48, 48, 12, 70, dict(src_dist=70.0, det_dist=140.0, det_spacing=1.7)),
         ("fanbeam", 40, 33, 7, 200, dict(src_dist=60.0, det_dist=120.0, det_spacing=0.5)),
         ("fanbeam", 64, 64, 8, 100, dict(src_dist=48.3, det_dist=80.0, det_spacing=2.0))]


@pytest.mark.parametrize("dt", ["float32", "float64"])
@pytest.mark.parametrize("value", [math.inf, math.nan])
@pytest.mark.parametrize("batch", [1, 2, 4, 5])
@pytest.mark.parametrize("geom", GEOMS)
def test_adjoint(geom, batch, value, dt):
    torch, api = require_gpu()
    kind, n1, n2, A, B, kw = geom
    ctx = api.Context(0)
    op = api.Operator(ctx, kind, n1, n2, dtype=getattr(torch, dt), n_angles=A, n_bins=B, **kw)
    rng = np.random.default_rng(A * B)
    s = rng.standard_normal((batch, A, B))
    e = np.zeros((A, B))
    k, m = int(rng.integers(A)), int(B // 2 + rng.integers(-B // 6, B // 6))
    s[batch // 2, k, m] = value
    e[k, m] = 1.0
    if kind == "radon":
        w = O.radon_adjoint(e, n1, n2, kw.get("angle_span", math.pi))
    else:
        w = O.fanbeam_adjoint(e, n1, n2, kw["src_dist"], kw["det_dist"], kw["det_spacing"])
    bad = ~np.isfinite(api.op_adjoint(op, torch.from_numpy(s).to(op.dtype).cuda()).double().cpu().numpy())
    for b in range(batch):
        if b != batch // 2:
            assert not bad[b].any()
    # a weight below the operator's rounding may be taken as zero or not
    tiny = 1e-6 if dt == "float32" else 1e-12
    assert bad[batch // 2][w > tiny].all()
    assert not bad[batch // 2][w == 0.0].any()
