"""Fan-beam forward on rays almost parallel to an axis, which leave the image
over many lines: every line that carries a weight is walked (float64 operators
to float64 rounding), and the pair agrees there."""
import math

import numpy as np
import pytest

import oracle.operators as O
from gpu_util import TOL, require_gpu

pytestmark = pytest.mark.gpu

# the ray (angle, bin) has slope about 1e-6 and grazes the image's edge within
# 3e-5 of a pixel over tens of lines; the others of its warp lie outside
N, A, B, R, D = 512, 720, 1025, 699.8585912999514, 731.1278000236199
ANGLE, BIN = 43, 800


@pytest.mark.parametrize("dt", ["f32", "f64"])
@pytest.mark.parametrize("batch", [1, 4])
def test_grazing_ray(dt, batch):
    torch, api = require_gpu()
    ctx = api.Context(0)
    op = api.Operator(ctx, "fanbeam", N, N, dtype=getattr(torch, {"f32": "float32", "f64": "float64"}[dt]),
                      n_angles=A, n_bins=B, src_dist=R, det_dist=D)
    x = torch.ones((batch, N, N), dtype=op.dtype, device="cuda")
    y = api.op_apply(op, x)[0, ANGLE].double().cpu().numpy()
    row, a, b, w = (t[ANGLE] for t in O.fanbeam_tables(N, N, A, B, R, D, 1.0))
    u = a[:, None] + b[:, None] * np.arange(N)[None, :]
    f = u - np.floor(u)
    inside = lambda p: (p >= 0) & (p < N)     # noqa: E731
    ref = w * (np.where(inside(np.floor(u)), 1.0 - f, 0.0) + np.where(inside(np.floor(u) + 1), f, 0.0)).sum(1)
    assert abs(b[BIN]) < 2e-6 and 0.0 < ref[BIN] < 0.1
    # float32: 512 samples of weights good to 2^-23
    assert abs(y[BIN] - ref[BIN]) <= (512 * 2.0 ** -23 if dt == "f32" else 1e-10)
    assert np.max(np.abs(y - ref)) <= TOL[dt] * np.max(ref)
    # the pair: <A 1, e_ray> = <1, A^T e_ray>
    s = torch.zeros((batch, A, B), dtype=op.dtype, device="cuda")
    s[:, ANGLE, BIN] = 1.0
    t = float(api.op_adjoint(op, s)[0].double().sum())
    assert abs(t - y[BIN]) <= (512 * 2.0 ** -22 if dt == "f32" else 1e-10)
