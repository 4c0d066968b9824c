"""The parallel-beam pair's interleaved lanes: batches cut into fours and rests,
mirror lanes (two for any shape, four for square images and even angle counts),
no mirror lanes (spans other than 180 degrees), ragged tiles, bins and angles,
against the float64 oracle."""
import math

import numpy as np
import pytest

import oracle.operators as O
from gpu_util import TOL, close, require_gpu

pytestmark = pytest.mark.gpu

# (n1, n2, angles, bins, span): tile edges at 32, warps of 32 and 64 bins, the
# orbits' ends (angle counts 1, 2, 3, multiples of 4 and not), detectors
# narrower than the image and wider than its diagonal
GEOMS = [
    (32, 32, 4, 46, math.pi),
    (33, 33, 6, 31, math.pi),
    (31, 31, 1, 33, math.pi),
    (40, 40, 2, 65, math.pi),
    (64, 64, 3, 97, math.pi),
    (17, 65, 8, 64, math.pi),
    (70, 37, 45, 90, math.pi),
    (48, 48, 10, 70, 2.0 * math.pi),
    (1, 5, 7, 9, math.pi),
    (96, 96, 180, 140, math.pi),
]


@pytest.fixture(scope="module")
def env():
    torch, api = require_gpu()
    return torch, api, api.Context(0)


@pytest.mark.parametrize("dt", ["f32", "f64"])
@pytest.mark.parametrize("geom", GEOMS)
@pytest.mark.parametrize("batch", [1, 2, 3, 4, 6, 33])
def test_pair_and_normal(env, geom, batch, dt):
    torch, api, ctx = env
    n1, n2, A, B, span = geom
    if batch == 33 and n1 * A > 2000:
        pytest.skip("one size of every kind is enough for the chunked batch")
    op = api.Operator(ctx, "radon", n1, n2, dtype=getattr(torch, {"f32": "float32", "f64": "float64"}[dt]),
                      n_angles=A, n_bins=B, angle_span=span)
    rng = np.random.default_rng(n1 * 1000 + A)
    x = rng.standard_normal((batch, n1, n2))
    s = rng.standard_normal((batch, A, B))
    t = lambda a: torch.from_numpy(a).to(op.dtype).cuda()      # noqa: E731
    fwd, adj = O.radon_apply(x, A, B, span), O.radon_adjoint(s, n1, n2, span)
    close(api.op_apply(op, t(x)), fwd, TOL[dt])
    close(api.op_adjoint(op, t(s)), adj, TOL[dt])
    close(api.op_normal(op, t(x)), O.radon_adjoint(fwd, n1, n2, span), TOL[dt])


@pytest.mark.parametrize("geom,ell", [((96, 96, 180, 140, math.pi), 32), ((70, 130, 200, 157, math.pi), 45),
                                      ((65, 64, 300, 130, 2.0 * math.pi), 41)])
def test_bf16_batch_in_eights(env, geom, ell):
    """The sketch's bf16 images, eight to a group (the last group of a chunk
    half full, or of fours and a rest): Y against the oracle on the stored
    Omega, within bf16's rounding of Y and the float32 operator's 1e-5."""
    torch, api, ctx = env
    n1, n2, A, B, span = geom
    op = api.Operator(ctx, "radon", n1, n2, dtype=torch.float32, n_angles=A, n_bins=B, angle_span=span)
    Om, Y = api.nys_sketch(ctx, op, ell, 3, store_dtype=torch.bfloat16)
    ref = O.radon_adjoint(O.radon_apply(Om.double().cpu().numpy(), A, B, span), n1, n2, span)
    err = np.abs(Y.double().cpu().numpy() - ref)
    assert np.all(err <= 2.0 ** -8 * np.abs(ref) + 1e-5 * np.abs(ref).max())
