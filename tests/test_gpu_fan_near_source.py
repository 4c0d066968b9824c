"""The fan-beam adjoint with the source beside the image: depths several times
apart within a 32 x 32 tile, where the bins that the nearest pixel needs lie
tens of pixels from the others, against the float64 oracle; and bins many
pixels apart."""
import math

import numpy as np
import pytest

import oracle.operators as O
from gpu_util import TOL, close, require_gpu

pytestmark = pytest.mark.gpu

# n1, n2, angles, bins, R - half diagonal, D, bin spacing
GEOMS = [(64, 64, 360, 100, 3.05, 80.0, 2.0), (40, 40, 72, 145, 2.05, 60.7, 1.0), (64, 64, 72, 123, 6.0, 102.5, 2.0),
         (96, 96, 72, 85, 3.0, 141.8, 4.0), (128, 128, 40, 240, 4.0, 189.0, 3.15), (33, 70, 72, 90, 12.0, 120.0, 2.5),
         (64, 64, 12, 5, 100.0, 300.0, 90.0), (64, 64, 24, 800, 2.5, 120.0, 0.4)]


@pytest.fixture(scope="module")
def env():
    torch, api = require_gpu()
    return torch, api, api.Context(0)


@pytest.mark.parametrize("dt", ["f32", "f64"])
@pytest.mark.parametrize("geom", GEOMS)
@pytest.mark.parametrize("batch", [1, 4])
def test_adjoint(env, geom, batch, dt):
    torch, api, ctx = env
    n1, n2, A, B, dR, D, du = geom
    R = 0.5 * math.hypot(n1, n2) + dR
    op = api.Operator(ctx, "fanbeam", n1, n2, dtype=getattr(torch, {"f32": "float32", "f64": "float64"}[dt]),
                      n_angles=A, n_bins=B, src_dist=R, det_dist=D, det_spacing=du)
    s = np.random.default_rng(n1 + A).standard_normal((batch, A, B))
    got = api.op_adjoint(op, torch.from_numpy(s).to(op.dtype).cuda())
    close(got, O.fanbeam_adjoint(s, n1, n2, R, D, du), TOL[dt])
