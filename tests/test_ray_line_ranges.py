"""Host-side check of the lines that the forward ray kernels walk, restated in
numpy (float32 as the kernels evaluate it).  A ray's position on line l is u = a
+ b l; every line with -1 < u < na carries a weight and must lie in the walked
range, for rays that cross the image's edge slowly above all (slope down to
1e-9, the crossing within 1e-7 of a pixel of the edge): a line left out is a
sample dropped silently."""
import math

import numpy as np
import pytest

f = np.float32


def fan_range(a1, b, nl, na):
    """fan_fwd, from 1 + a and b in float32."""
    a0 = np.floor(a1)
    with np.errstate(divide="ignore", invalid="ignore"):
        e1, e2 = (f(-1) - a0) / b, (f(na + 2) - a0) / b
    lo = np.maximum(f(0), np.floor(np.fmin(e1, e2)) - f(2))
    hi = np.minimum(f(nl), np.ceil(np.fmax(e1, e2)) + f(3))
    steep = np.abs(b) * f(nl) > f(1)
    lo = np.where(steep, lo, 0).astype(np.int64)
    hi = np.where(steep, hi, np.where((a0 < f(-5)) | (a0 > f(na + 5)), 0, nl)).astype(np.int64)
    return lo, hi


@pytest.mark.parametrize("nl,na", [(512, 512), (2048, 100), (37, 64), (8192, 8192)])
@pytest.mark.parametrize("dt", ["f32", "f64"])
def test_fan_rays(nl, na, dt):
    rng = np.random.default_rng(nl + na)
    n = 4000
    b = rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-9.0, 0.0, n)
    # the ray is at one of the edges, and some 1e-7 .. 1 pixels off, on line l0
    l0 = rng.uniform(-2.0, nl + 2.0, n)
    a = rng.choice([-1.0, float(na)], n) + rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-7.0, 0.0, n) - b * l0
    if dt == "f32":
        q, bq = np.rint((1.0 + a) * 2.0 ** 40).astype(np.int64), np.rint(b * 2.0 ** 40).astype(np.int64)
        a, b = q * 2.0 ** -40 - 1.0, bq * 2.0 ** -40
    lo, hi = fan_range((1.0 + a).astype(f), b.astype(f), nl, na)
    u = a[:, None] + b[:, None] * np.arange(nl)[None, :]
    live = (u > -1.0) & (u < na)
    l = np.arange(nl)[None, :]
    assert live.any() and not (live & ((l < lo[:, None]) | (l >= hi[:, None]))).any()


@pytest.mark.parametrize("n1,n2,B", [(512, 512, 736), (2048, 96, 2100), (96, 2048, 2100), (64, 64, 300), (40, 33, 20_000), (32, 40, 12_600_001),
                                     (32, 32, 60_000_000)])
@pytest.mark.parametrize("CB", [1, 2])
def test_parallel_warps(n1, n2, B, CB):
    """radon_fwd: a warp's 32 CB bins share a range, from the whole positions of
    its first and last bin on line 0."""
    ths = [s * math.pi / 2 + d for s in (0, 1, 2) for d in (0.0, 3e-8, 2e-6, 1.3e-5, 4e-4, 0.02, -3e-8, -2e-6, -0.3)]
    for th in ths + [0.25 * math.pi, 0.7]:
        cs, sn = math.cos(th), math.sin(th)
        rs = abs(cs) + 1e-9 >= abs(sn)
        (nl, na), (den, oth) = ((n1, n2), (cs, sn)) if rs else ((n2, n1), (sn, cs))
        cq, invh, th2 = (int(np.rint(v * 2.0 ** 40)) for v in ((na + 1) / 2, 0.5 / den, 0.5 * oth / den))
        u0q, invq, tq = cq - (B - 1) * invh + (nl - 1) * th2, 2 * invh, 2 * th2
        far = n1 + n2 + 64
        m_lo, m_hi = max(0, (B - 1 - far) // 2), min(B - 1, (B - 1 + far) // 2)

        def at(m, l):      # 64-bit integers that wrap
            p = (u0q + np.asarray(m, object) * invq - np.asarray(l, object) * tq + 2 ** 63) % 2 ** 64 - 2 ** 63
            return p.astype(np.int64) if isinstance(p, np.ndarray) else p

        tl = f(tq) * f(2.0 ** -40)
        step = 32 * CB
        starts = range(0, B, step)
        if B > 100_000:       # around the image, where positions wrap round onto it, and the ends
            mids = [B // 2 + s * int(2 ** 24 * abs(den)) for s in (-1, 0, 1)] + [0, B - 1]
            starts = sorted({(m // step + d) * step for m in mids for d in range(-4, 5) if 0 <= (m // step + d) * step < B})
        for m0 in starts:
            m1 = min(m0 + 32 * CB - 1, B - 1)
            qa, qb = (f((at(m, 0) >> 40) - 1) for m in (m0, m1))
            qmin, qmax = min(qa, qb), max(qa, qb) + f(1)
            lo, hi = 0, nl
            if abs(tl) > f(1e-6):
                e1, e2 = (qmin - f(na)) / tl, (qmax + f(1)) / tl
                lo = int(max(f(0), np.floor(min(e1, e2)) - f(2)))
                hi = int(min(f(nl), np.ceil(max(e1, e2)) + f(3)))
            elif qmax < -3 or qmin > na + 2:
                hi = 0
            if m0 > m_hi or m0 + 32 * CB <= m_lo:
                hi = 0
            m, l = np.arange(m0, m1 + 1)[:, None], np.arange(nl)[None, :]
            u = ((u0q + m * np.int64(invq) - l * np.int64(tq)) if abs(u0q) < 2 ** 62 else at(m, l)) * 2.0 ** -40 - 1.0
            exact = (na - 1) / 2 + (m - (B - 1) / 2) / den - (l - (nl - 1) / 2) * (oth / den)
            seen = (exact > -1.0) & (exact < na)
            assert np.all(np.abs(u - exact)[seen] <= 2.0 ** -40 * far)
            walked = (l >= lo) & (l < hi)
            assert not (walked & (u > -1.0 + 1e-6) & (u < na - 1e-6) & ~seen).any()
            assert not (seen & ((l < lo) | (l >= hi))).any()
