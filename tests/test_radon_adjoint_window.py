"""Host-side check of the parallel-beam adjoint's positions, restated in numpy: the
fixed-point position of every pixel of a 32 x 32 tile stays inside the 48
staged bins (its two bins are index and index + 1), the bins either side of the
pixel's exact position are those two to rounding, the position being good to
2^-26 of a bin (float32 operators) whatever the angle, the tile and the size of
the image."""
import math

import numpy as np
import pytest

ATS, AWIN = 32, 48


def positions(n1, n2, B, th, i0, j0, bits):
    """(index, fraction) of the tile's pixels and the first staged bin (from the middle
    bin (B - 1) // 2 on)."""
    cs, sn = math.cos(th), math.sin(th)
    m00 = cs * (j0 - 0.5 * (n2 - 1)) + (sn * (i0 - 0.5 * (n1 - 1)) + 0.5 * ((B - 1) & 1))
    lo = math.floor(m00 + min(0.0, (ATS - 1) * cs) + min(0.0, (ATS - 1) * sn) - 1e-3)
    tx, ty = np.meshgrid(np.arange(ATS), np.arange(ATS))
    if bits == 32:
        p0 = int(np.rint((m00 + 16 * (cs + sn) - lo) * 2.0 ** 32))
        dj, di = int(np.rint(cs * 2.0 ** 30)), int(np.rint(sn * 2.0 ** 30))
        assert abs(dj) <= 2 ** 30 and abs(di) <= 2 ** 30
        p = p0 + (((tx - 16) * dj + (ty - 16) * di) << 2)
        return p >> 32, (p & 0xffffffff) * 2.0 ** -32, lo, tx, ty
    p0 = int(np.rint((m00 + 16 * (cs + sn) - lo) * 2.0 ** 57)) + 16
    dj, di = int(np.rint(cs * 2.0 ** 57)), int(np.rint(sn * 2.0 ** 57))
    p = np.array([[p0 + (int(x) - 16) * dj + (int(y) - 16) * di for x in range(ATS)] for y in range(ATS)], dtype=object)
    assert p.min() >= 0 and p.max() < 2 ** 64
    return (p >> 57).astype(np.int64), ((p & (2 ** 57 - 1)) * 2.0 ** -57).astype(np.float64), lo, tx, ty


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("n1,n2,B", [(512, 512, 736), (4096, 4096, 5794), (33, 70, 64), (6000, 40, 700), (1, 1, 1)])
def test_positions(n1, n2, B, bits):
    rng = np.random.default_rng(n1 + B)
    ths = [k * math.pi / 4 for k in range(8)] + [math.nextafter(math.pi / 4, 0), 1e-9] + list(rng.uniform(0, 2 * math.pi, 25))
    tiles = [(0, 0), ((n1 - 1) // ATS * ATS, (n2 - 1) // ATS * ATS), (n1 // 2 // ATS * ATS, 0)]
    for th in ths:
        for i0, j0 in tiles:
            idx, frac, lo, tx, ty = positions(n1, n2, B, th, i0, j0, bits)
            assert idx.min() >= 0 and idx.max() + 1 < AWIN
            ld = np.longdouble
            cs, sn = np.cos(ld(th)), np.sin(ld(th))
            m = cs * (j0 + tx - ld(n2 - 1) / 2) + sn * (i0 + ty - ld(n1 - 1) / 2) + ld((B - 1) & 1) / 2
            err = np.abs((lo + idx) + ld(1) * frac - m)
            # float64 rounding of the first pixel's position, then the fixed point
            assert np.max(err) <= (2.0 ** -26 if bits == 32 else 2.0 ** -48) + 4 * np.finfo(float).eps * (n1 + n2)
