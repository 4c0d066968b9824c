"""Host-side check of the fan-beam adjoint's candidate bins, restated in numpy
(float32 geometry as the kernel evaluates it, float64 ray tables as the host
builds them).  For every pixel of a 32 x 32 tile and every segment of bins that
reaches the tile:

* the walked bins (K from a common start, or the pixel's own first and last bin
  where K is 0) hold every bin whose ray passes within one pixel of the pixel
  along the segment's kind of line -- another one would be dropped silently;
* the offset of every walked bin's ray, taken modulo 32 pixels (float32
  operators) or 512 (float64), gives the weight of the offset itself -- a ray
  32 pixels away would come back with a weight near one.

Sources right beside the image, where a tile's depths are several times apart,
are the hard ones; the large images are sampled at a few tiles."""
import math

import numpy as np
import pytest

import oracle.operators as O

f = np.float32
ATS, AWIN, AKMAX = 32, 192, 64


def segments(rs, up):
    out, m, B = [], 0, len(rs)
    while m < B:
        e = m + 1
        while e < B and rs[e] == rs[m] and up[e] == up[m]:
            e += 1
        out.append((m, e, bool(rs[m]), (1 if up[m] else -1) * (1 if rs[m] else -1)))
        m = e
    return out


def int_bits(du, R, D, n1, n2, bits):
    spacing = math.sqrt(2.0) * du * (R + 0.5 * math.hypot(n1, n2) + 2.0) / D
    ib = 9 if bits == 64 else 5
    while ib < 25 and 2.0 ** ib < 8.0 + 0.05 * spacing:
        ib += 1
    return ib


def tile_job(n1, n2, B, R, G, e, seg, i0, j0, reach):
    """The job of a segment on a tile: None when it does not reach the tile."""
    lo, hi, rs, sgn = seg
    ex, ey = e
    px, py = f(j0) - f(0.5) * f(n2 - 1), f(i0) - f(0.5) * f(n1 - 1)
    a0, d0 = -px * ey + py * ex, R - (px * ex + py * ey)
    ar, ap, dr, dp = (ex, -ey, -ey, -ex) if rs else (-ey, ex, -ex, -ey)
    ti, tj = f(min(ATS, n1 - i0) - 1), f(min(ATS, n2 - j0) - 1)
    tr, tp = (ti, tj) if rs else (tj, ti)
    sf, cb = f(sgn), f(0.5) * f(B - 1)
    r, p = np.array([0, 1, 0, 1], f) * tr, np.array([0, 0, 1, 1], f) * tp
    a, d = a0 + ar * r + ap * p, d0 + dr * r + dp * p
    ml, mh = cb + G * (a - sf * ap) / (d - sf * dp), cb + G * (a + sf * ap) / (d + sf * dp)
    if not (ml.min() < f(hi) + 1 and mh.max() > f(lo) - 1):
        return None
    d_min, d_max, num = (d - abs(dp)).min(), (d + abs(dp)).max(), np.abs(ap * d - a * dp)
    terms = abs(px) + abs(py) + f(64)
    eps = f(0.01) + f(2.0 ** -21) * (G / d_min) * (terms + (np.abs(a).max() / d_min) * (R + terms))
    K = int(min(f(2) * G * num.max() / (d_min * d_min) + f(4) * eps, f(1e6))) + 1
    mlo = int(np.floor(ml.min() - eps)) - 1
    wn = int(np.ceil(max(ml.max() + eps + f(K), mh.max()))) + 2 - mlo
    Kd = f(K) * d_max
    if wn > AWIN or K > AKMAX or not (Kd * d_max < reach * (G * num.min() - Kd * abs(dp))):
        K = 0
    return dict(a0=a0, d0=d0, ar=ar, ap=ap, dr=dr, dp=dp, tr=int(tr), tp=int(tp), sf=sf, mlo=mlo, wn=wn, K=K, eps=eps,
                mc=cb - f(mlo))


def check(n1, n2, A, B, R, D, du, angles, bits, tiles=None):
    row, a, b, _ = O.fanbeam_tables(n1, n2, A, B, R, D, du)
    th = np.arange(A) * (2.0 * math.pi / A)
    um = (np.arange(B) - (B - 1) / 2.0) * du
    mod = 2.0 ** int_bits(du, R, D, n1, n2, bits)
    G, Rf = f(D / du), f(R)
    walked = dropped = wrapped = fast = slow = 0
    tiles = tiles or [(i, j) for i in range(0, n1, ATS) for j in range(0, n2, ATS)]
    for k in angles:
        cs, sn = math.cos(th[k]), math.sin(th[k])
        up = np.where(row[k], -D * sn + um * cs, -D * cs - um * sn) > 0
        for seg in segments(row[k], up):
            lo, hi, rs, _ = seg
            for i0, j0 in tiles:
                J = tile_job(n1, n2, B, Rf, G, (f(cs), f(sn)), seg, i0, j0, f(mod) - f(2))
                rr, pp = np.meshgrid(np.arange(min(ATS, (n1 - i0) if rs else (n2 - j0))),
                                     np.arange(min(ATS, (n2 - j0) if rs else (n1 - i0))), indexing="ij")
                # the bins looked at: the window and 40 more either side
                m0, m1 = (lo, hi) if J is None else (max(lo, J["mlo"] - 40), min(hi, J["mlo"] + J["wn"] + 40))
                m = np.arange(m0, max(m0, m1))
                off = a[k, m] + b[k, m] * (rr + (i0 if rs else j0))[..., None] - (pp + (j0 if rs else i0))[..., None]
                touch = np.abs(off) < 1.0 - 1e-12
                if J is None:
                    dropped += int(touch.sum())
                    continue
                fr = rr.astype(f)
                if J["K"]:
                    fast += 1
                    fp = pp.astype(f) - J["sf"]
                    mm = J["mc"] + G * ((J["a0"] + J["ar"] * fr + J["ap"] * fp) / (J["d0"] + J["dr"] * fr + J["dp"] * fp))
                    c0 = np.maximum(0, np.minimum(np.ceil(mm - J["eps"]).astype(np.int64), J["wn"] - J["K"]))
                    c1 = c0 + J["K"] - 1
                else:
                    slow += 1
                    aa = J["a0"] + J["ar"] * fr + J["ap"] * pp.astype(f)
                    dd = J["d0"] + J["dr"] * fr + J["dp"] * pp.astype(f)
                    ml = J["mc"] + G * ((aa - J["sf"] * J["ap"]) / (dd - J["sf"] * J["dp"]))
                    mh = J["mc"] + G * ((aa + J["sf"] * J["ap"]) / (dd + J["sf"] * J["dp"]))
                    c0 = np.maximum(np.ceil(ml - J["eps"]), 0).astype(np.int64)
                    c1 = np.minimum(np.floor(mh + J["eps"]), J["wn"] - 1).astype(np.int64)
                on = (m >= J["mlo"] + c0[..., None]) & (m <= J["mlo"] + c1[..., None])
                dropped += int((touch & ~on).sum())
                w = (off + mod / 2) % mod - mod / 2
                wrapped += int((on & (np.abs(off) >= 1.0) & (np.abs(w) < 1.0 - 1e-9)).sum())
                walked += int((on & touch).sum())
    return walked, dropped, wrapped, fast, slow


# n1, n2, angles, bins, R - half diagonal, D, bin spacing
NEAR = [(64, 64, 360, 100, 3.05, 80.0, 2.0), (40, 40, 72, 145, 2.05, 60.7, 1.0), (64, 64, 72, 123, 6.0, 102.5, 2.0),
        (96, 96, 72, 85, 3.0, 141.8, 4.0), (128, 128, 72, 240, 4.0, 189.0, 3.15), (33, 70, 72, 90, 12.0, 120.0, 2.5),
        (64, 64, 72, 800, 2.5, 120.0, 0.4), (200, 200, 72, 300, 25.0, 400.0, 3.0)]


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("geom", NEAR)
def test_source_beside_the_image(geom, bits):
    n1, n2, A, B, dR, D, du = geom
    R = 0.5 * math.hypot(n1, n2) + dR
    walked, dropped, wrapped, _, slow = check(n1, n2, A, B, R, D, du, [0, A // 8, 65 * A // 360], bits)
    assert walked > 0 and dropped == 0 and wrapped == 0
    assert slow > 0 or dR > 3      # the hard tiles do leave the common walk


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("geom", [(64, 64, 12, 11, 30.0, 150.0, 20.0), (64, 64, 12, 5, 100.0, 300.0, 90.0),
                                  (96, 50, 9, 2000, 60.0, 250.0, 0.2), (1, 5, 2, 9, 3.5, 12.0, 1.0)])
def test_sparse_and_dense_bins(geom, bits):
    n1, n2, A, B, dR, D, du = geom
    R = 0.5 * math.hypot(n1, n2) + dR
    walked, dropped, wrapped, _, _ = check(n1, n2, A, B, R, D, du, range(A), bits)
    assert walked > 0 and dropped == 0 and wrapped == 0


def test_usual_geometry_stays_on_the_common_walk():
    walked, dropped, wrapped, fast, slow = check(512, 512, 720, 1024, 700.0, 1400.0, 1.2, [0, 45, 90, 133], 32,
                                                 [(0, 0), (224, 256), (480, 480), (480, 0)])
    assert walked > 0 and dropped == 0 and wrapped == 0 and slow == 0 and fast > 0


@pytest.mark.parametrize("n,bits", [(2048, 32), (2048, 64), (8192, 64)])
@pytest.mark.parametrize("near", [False, True])
def test_large_images(n, bits, near):
    """Float rounding of the geometry grows with the image; eps grows with it."""
    R = 0.5 * math.hypot(n, n) + (3.0 if near else 0.5 * n)
    du = 0.6 * R / n if not near else 2.0
    B = 4 * n
    t = n // 2
    walked, dropped, wrapped, _, _ = check(n, n, 360, B, R, 2.0 * R, du, [3, 45, 130], bits,
                                           [(0, 0), (t, t), (n - ATS, n - ATS), (n - ATS, 0), (t, n - ATS)])
    assert walked > 0 and dropped == 0 and wrapped == 0
