"""The fan-beam pair's interleaved lanes: batches cut into fours and rests,
mirror lanes (four with an even number of angles over a full circle, two with
an odd one), none over other spans, odd bin counts whose central ray runs at 45
degrees, bins denser than the adjoint's staged window and coarser than pixels,
a source just outside the image, against the float64 oracle."""
import math

import numpy as np
import pytest

import oracle.operators as O
from gpu_util import TOL, close, require_gpu

pytestmark = pytest.mark.gpu

# (n1, n2, angles, bins, span, R, D, du)
GEOMS = [
    (32, 32, 8, 47, 2.0 * math.pi, 60.0, 120.0, 1.5),       # angles at 45 degrees, a bin on the central ray
    (33, 31, 7, 64, 2.0 * math.pi, 50.0, 100.0, 1.3),       # two lanes
    (40, 65, 10, 90, 2.0 * math.pi, 90.0, 170.0, 1.7),
    (64, 64, 3, 97, math.pi, 100.0, 180.0, 1.5),            # no symmetry used
    (24, 24, 4, 700, 2.0 * math.pi, 40.0, 80.0, 0.1),       # windows of several pieces
    (48, 48, 12, 11, 2.0 * math.pi, 70.0, 150.0, 20.0),     # bins many pixels apart
    (20, 20, 16, 33, 2.0 * math.pi, 16.5, 40.0, 2.5),       # the source next to the corner
    (1, 5, 2, 9, 2.0 * math.pi, 6.0, 12.0, 1.0),
]


@pytest.fixture(scope="module")
def env():
    torch, api = require_gpu()
    return torch, api, api.Context(0)


@pytest.mark.parametrize("dt", ["f32", "f64"])
@pytest.mark.parametrize("geom", GEOMS)
@pytest.mark.parametrize("batch", [1, 3, 6])
def test_pair_and_normal(env, geom, batch, dt):
    torch, api, ctx = env
    n1, n2, A, B, span, R, D, du = geom
    op = api.Operator(ctx, "fanbeam", n1, n2, dtype=getattr(torch, {"f32": "float32", "f64": "float64"}[dt]),
                      n_angles=A, n_bins=B, angle_span=span, src_dist=R, det_dist=D, det_spacing=du)
    rng = np.random.default_rng(n1 * 1000 + A)
    x = rng.standard_normal((batch, n1, n2))
    s = rng.standard_normal((batch, A, B))
    t = lambda a: torch.from_numpy(a).to(op.dtype).cuda()      # noqa: E731
    fwd = O.fanbeam_apply(x, A, B, R, D, du, span)
    close(api.op_apply(op, t(x)), fwd, TOL[dt])
    close(api.op_adjoint(op, t(s)), O.fanbeam_adjoint(s, n1, n2, R, D, du, span), TOL[dt])
    close(api.op_normal(op, t(x)), O.fanbeam_adjoint(fwd, n1, n2, R, D, du, span), TOL[dt])
