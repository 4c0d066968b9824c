"""The weights of the float32 ray transforms, read off one by one: a ray meets a
pixel in one sample, so the transform of an image with a single pixel returns
single weights.  They are held to a few roundings of 2^-24 for images of any
size (positions are carried in more bits than the weights); the adjoint of a
sinogram with one bin an angle likewise."""
import math

import numpy as np
import pytest

import oracle.operators as O
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def pixels(n, count):
    rng = np.random.default_rng(n)
    return [(n - 1, n - 1), (0, n - 1), (n // 2, 3)] + [tuple(int(v) for v in rng.integers(0, n, 2)) for _ in range(count)]


def parallel(torch, api, n):
    """Operator and the weights (angles, bins) of a pixel in 64 bits."""
    A, B, span = 14, int(1.45 * n), 2.6
    op = api.Operator(api.Context(0), "radon", n, n, dtype=torch.float32, n_angles=A, n_bins=B, angle_span=span)
    c, t = (n - 1) / 2.0, np.arange(B) - (B - 1) / 2.0

    def weights(i, j):
        out = np.zeros((A, B))
        for k in range(A):
            cs, sn = math.cos(k * (span / A)), math.sin(k * (span / A))
            rs = abs(cs) + 1e-9 >= abs(sn)
            den, oth, line, pos = (cs, sn, i, j) if rs else (sn, cs, j, i)
            out[k] = np.maximum(0.0, 1.0 - np.abs(c + t / den - (line - c) * (oth / den) - pos)) / abs(den)
        return out
    return op, weights


def fan(torch, api, n):
    A, B, R, D, span = 9, 2 * n, 1.3 * n, 2.2 * n, 5.0
    op = api.Operator(api.Context(0), "fanbeam", n, n, dtype=torch.float32, n_angles=A, n_bins=B, angle_span=span,
                      src_dist=R, det_dist=D)
    row, a, b, w = O.fanbeam_tables(n, n, A, B, R, D, 1.0, span)

    def weights(i, j):
        return w * np.maximum(0.0, 1.0 - np.abs(a + b * np.where(row, i, j) - np.where(row, j, i)))
    return op, weights


@pytest.mark.parametrize("geom,n", [(parallel, 512), (parallel, 2048), (parallel, 4096), (fan, 512), (fan, 2048)])
@pytest.mark.parametrize("batch", [1, 4])
def test_forward(geom, n, batch):
    torch, api = require_gpu()
    op, weights = geom(torch, api, n)
    err = []
    for i, j in pixels(n, 5):
        x = torch.zeros((batch, n, n), device="cuda")
        x[:, i, j] = 1.0
        y = api.op_apply(op, x)[batch - 1].double().cpu().numpy()
        ref = weights(i, j)
        assert np.all(np.abs(y[ref == 0.0]) <= 2.0 * U)
        err.append((y - ref)[ref > 0.0])
    err = np.concatenate(err)
    # the fraction and one less it (U / 2 each), 1 / |den| <= 1.415 and the product (U each)
    assert np.max(np.abs(err)) <= 1.415 * 3.0 * U
    assert np.sqrt(np.mean(err ** 2)) <= U


@pytest.mark.parametrize("n", [512, 2048, 4096])
@pytest.mark.parametrize("batch", [1, 4])
def test_parallel_adjoint(n, batch):
    torch, api = require_gpu()
    op, weights = parallel(torch, api, n)
    A, B = op.meas_shape
    err = []
    for i, j in pixels(n, 9):
        ref = weights(i, j)
        for k in range(A):
            for m in np.nonzero(ref[k])[0]:
                s = torch.zeros((batch, A, B), device="cuda")
                s[:, k, m] = 1.0
                err.append(float(api.op_adjoint(op, s)[batch - 1, i, j]) - ref[k, m])
    err = np.array(err)
    # 1 / |den| and its difference to 1 / den^2 <= 2, 1 / den^2 itself, the fraction
    # (U / 2, times 1 / den^2) and the sum: U each
    assert np.max(np.abs(err)) <= 4.0 * U
    assert np.sqrt(np.mean(err ** 2)) <= U


@pytest.mark.parametrize("n,B,du", [(512, 1024, 1.0), (2048, 4096, 1.0), (512, 200, 12.0), (512, 60, 40.0)])
def test_fan_adjoint(n, B, du):
    """Bins of half a pixel to 40 pixels: the offsets keep their fraction bits."""
    torch, api = require_gpu()
    A, R, D, span = 9, 1.3 * n, 2.2 * n, 5.0
    op = api.Operator(api.Context(0), "fanbeam", n, n, dtype=torch.float32, n_angles=A, n_bins=B, angle_span=span,
                      src_dist=R, det_dist=D, det_spacing=du)
    row, a, b, w = O.fanbeam_tables(n, n, A, B, R, D, du, span)
    err = []
    for i, j in pixels(n, 20):
        ref = w * np.maximum(0.0, 1.0 - np.abs(a + b * np.where(row, i, j) - np.where(row, j, i)))
        for k in range(A):
            for m in np.nonzero(ref[k])[0]:
                s = torch.zeros((1, A, B), device="cuda")
                s[:, k, m] = 1.0
                err.append((float(api.op_adjoint(op, s)[0, i, j]) - ref[k, m]) / w[k, m])
    # the offset (2^-28, and as much 16 times from the slope), its conversion and one
    # less it (U / 2 each), the ray's weight and the product (U each)
    assert np.max(np.abs(err)) <= 4.1 * U
    assert np.sqrt(np.mean(np.square(err))) <= U
