"""The weights of the float32 ray transforms, read off one by one: a row-step (or
column-step) ray meets a pixel in one sample, so the transform of an image of
isolated pixels, and the adjoint of isolated bins, return single weights.  They
are held to a few roundings of 2^-24 for images of any size (positions are
carried in more bits than the weights)."""
import math

import numpy as np
import pytest

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def exact_weights(n, B, th, i, j):
    """Row of the transform's weights of pixel (i, j) over the bins, 64 bits."""
    cs, sn = math.cos(th), math.sin(th)
    c, cb = (n - 1) / 2.0, (B - 1) / 2.0
    rs = abs(cs) + 1e-9 >= abs(sn)
    den, oth = (cs, sn) if rs else (sn, cs)
    line, pos = (i, j) if rs else (j, i)
    u = c + (np.arange(B) - cb) / den - (line - c) * (oth / den)
    return np.maximum(0.0, 1.0 - np.abs(u - pos)) / abs(den)


@pytest.mark.parametrize("n", [512, 2048, 4096])
@pytest.mark.parametrize("batch", [1, 4])
def test_parallel_beam(n, batch):
    torch, api = require_gpu()
    ctx = api.Context(0)
    A, B = 14, int(1.45 * n)
    op = api.Operator(ctx, "radon", n, n, dtype=torch.float32, n_angles=A, n_bins=B, angle_span=2.6)
    rng = np.random.default_rng(n)
    pix = [(n - 1, n - 1), (0, n - 1), (n // 2, 3)] + [tuple(rng.integers(0, n, 2)) for _ in range(3)]
    ef, ea = [], []
    for i, j in pix:
        x = torch.zeros((batch, n, n), device="cuda")
        x[:, i, j] = 1.0
        y = api.op_apply(op, x)[batch - 1].double().cpu().numpy()
        ref = np.stack([exact_weights(n, B, k * (2.6 / A), i, j) for k in range(A)])
        hit = ref > 0.0
        ef.append((y - ref)[hit])
        assert np.all(np.abs(y)[~hit] <= 2 * U)
        # one bin per angle, the one nearest to the pixel's centre or its neighbour
        s = torch.zeros((batch, A, B), device="cuda")
        for k in range(A):
            m = np.nonzero(hit[k])[0]
            m = int(m[rng.integers(m.size)])
            s.zero_()
            s[:, k, m] = 1.0
            got = float(api.op_adjoint(op, s)[batch - 1, i, j])
            ea.append(got - ref[k, m])
    ef, ea = np.concatenate(ef), np.array(ea)
    # forward: the fraction (1/2 U), 1 - f (1/2), 1/|den| <= 1.415 and the product (1 each)
    assert np.max(np.abs(ef)) <= 1.415 * 3.0 * U and np.sqrt(np.mean(ef ** 2)) <= U
    # adjoint: the constants 1/|den| and 1/den^2 <= 2 (2 U), the fraction times 1/den^2 (1), the sum (1)
    assert np.max(np.abs(ea)) <= 4.0 * U and np.sqrt(np.mean(ea ** 2)) <= 1.4 * U


@pytest.mark.parametrize("n", [512, 2048])
def test_fan_beam(n):
    import oracle.operators as O
    torch, api = require_gpu()
    ctx = api.Context(0)
    A, B, R, D = 9, 2 * n, 1.3 * n, 2.2 * n
    op = api.Operator(ctx, "fanbeam", n, n, dtype=torch.float32, n_angles=A, n_bins=B, angle_span=5.0, src_dist=R,
                      det_dist=D)
    row, a, b, w = O.fanbeam_tables(n, n, A, B, R, D, 1.0, 5.0)
    rng = np.random.default_rng(n)
    ef, ea = [], []
    for i, j in [(n - 1, n - 1), (n // 2, 3)] + [tuple(rng.integers(0, n, 2)) for _ in range(4)]:
        u = a + b * np.where(row, i, j)
        ref = w * np.maximum(0.0, 1.0 - np.abs(u - np.where(row, j, i)))
        x = torch.zeros((1, n, n), device="cuda")
        x[:, i, j] = 1.0
        y = api.op_apply(op, x)[0].double().cpu().numpy()
        hit = ref > 0.0
        ef.append((y - ref)[hit])
        for k in range(A):
            m = np.nonzero(hit[k])[0]
            m = int(m[rng.integers(m.size)])
            s = torch.zeros((1, A, B), device="cuda")
            s[:, k, m] = 1.0
            ea.append(float(api.op_adjoint(op, s)[0, i, j]) - ref[k, m])
    ef, ea = np.concatenate(ef), np.array(ea)
    assert np.max(np.abs(ef)) <= 1.415 * 3.0 * U and np.sqrt(np.mean(ef ** 2)) <= U
    # adjoint: offsets in 27 fraction bits, the slope's rounding up to 31 times
    assert np.max(np.abs(ea)) <= 1.415 * 5.0 * U and np.sqrt(np.mean(ea ** 2)) <= 1.5 * U
