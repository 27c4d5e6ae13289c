"""The tile forward's unchecked batches, emulated in float32 on the CPU.

The forward walks a ray's bands in batches of four and loads a batch without
per-band bounds tests when the lower pixels m0 of its first and last band both lie
in [0, n_minor - 2]: m0 is monotone in the band, so the two between lie there too,
and so does every upper pixel m0 + 1.  Over every ray and band-chunk count of
several geometries this checks that m0 is monotone and that no band of an admitted
batch has a pixel outside the image.

The band point is two fused multiply-adds, emulated by FP64 products and sums
rounded once to FP32, which may be one ulp off in rare ties.  The second test covers
that: for every view and image a plan takes (at most 1024 views, 16384 pixels), a
band moves the point by many ulps of its largest value, so rounding cannot reverse
two bands.
"""
import math

import numpy as np
import pytest

f32 = np.float32


def _fma(a, b, c):
    return (np.asarray(a, np.float64) * np.asarray(b, np.float64) + np.asarray(c, np.float64)).astype(f32)


def _snap(x):
    return float(round(x)) if abs(x - round(x)) < 1e-12 else x


def _slope(i, na):
    c, s = _snap(math.cos(i * math.pi / na)), _snap(math.sin(i * math.pi / na))
    col = abs(c) < abs(s)
    cm, cn = (s, c) if col else (c, s)
    return col, cm, cn


def _batches(nx, ny, na, nb, pixel_mm, bin_mm, views, chunk_counts):
    """(admitted, out of bounds, not monotone) over the batches of the views' rays."""
    admitted = outside = reversed_ = 0
    for i in views:
        col, cm, cn = _slope(i, na)
        n_minor, n_major = (ny, nx) if col else (nx, ny)
        du64 = -cn / cm
        du = f32(du64)
        du_lo = f32(du64 - float(du))
        inv_du = f32(-cm / cn) if cn != 0.0 else f32(0.0)
        u = (np.arange(nb) - 0.5 * (nb - 1)) * bin_mm / (cm * pixel_mm) + (0.5 if n_minor % 2 else 0.0)
        ui_f = np.rint(u)
        ux, uy = ui_f.astype(f32), (u - ui_f).astype(f32)
        mo, hm = n_minor >> 1, f32(0.5 * n_major)
        uc = (ux + uy).astype(f32)
        if du == 0.0:
            k_lo = np.zeros(nb, np.int64)
            k_hi = np.where((uc >= f32(-mo)) & (uc < f32(n_minor - mo)), n_major, 0)
        else:
            ka = _fma((f32(-mo - 1) - uc).astype(f32), inv_du, hm)
            kb = _fma((f32(n_minor - mo + 1) - uc).astype(f32), inv_du, hm)
            kmax = f32(n_major + 1)
            lo = np.minimum(np.maximum(np.minimum(ka, kb), f32(-1)), kmax)
            hi = np.maximum(np.minimum(np.maximum(ka, kb), kmax), f32(-1))
            k_lo = np.maximum(0, np.floor(lo).astype(np.int64) - 1)
            k_hi = np.minimum(n_major, np.ceil(hi).astype(np.int64) + 1)
        # every band's lower pixel, [band, ray]
        kc = (np.arange(n_major + 1).astype(f32) - hm).astype(f32)[:, None]
        point = _fma(kc, du, _fma(kc, du_lo, uy[None, :]))
        m0 = np.floor(np.minimum(point[:-1], point[1:])).astype(np.int64) + (ux.astype(np.int64) + mo)
        step = np.diff(m0, axis=0)
        reversed_ += int((step < 0).sum() if du >= 0 else (step > 0).sum())
        rays = np.arange(nb)
        for chunks in chunk_counts:
            per = (n_major + chunks - 1) // chunks
            for ch in range(chunks):
                first = np.maximum(k_lo, ch * per)
                last = np.minimum(k_hi, (ch + 1) * per)
                for start in range(0, per, 4):
                    k = first + start
                    whole = k + 4 <= last
                    r, k = rays[whole], k[whole]
                    ends = [m0[k + b, r] for b in range(4)]
                    ok = [(m >= 0) & (m <= n_minor - 2) for m in ends]
                    admit = ok[0] & ok[3]
                    admitted += int(admit.sum())
                    outside += int((admit & ~(ok[1] & ok[2])).sum())
    return admitted, outside, reversed_


@pytest.mark.parametrize("nx,ny,na,nb,pixel_mm,bin_mm,every", [
    (64, 64, 60, 91, 2.0, 2.0, 1), (37, 29, 23, 41, 1.7, 1.3, 1), (128, 128, 90, 183, 2.0, 2.0, 1),
    (96, 80, 37, 131, 2.0, 1.6, 1), (256, 256, 180, 367, 2.0, 2.0, 6), (3, 64, 1024, 15, 2.0, 2.0, 8),
    (300, 7, 1024, 33, 2.0, 2.0, 16), (2, 50, 31, 9, 2.0, 1.0, 1), (1, 40, 20, 5, 2.0, 1.0, 1)])
def test_unchecked_batches_stay_inside_the_image(nx, ny, na, nb, pixel_mm, bin_mm, every):
    # every view next to an axis, and a sample of the others
    views = sorted(set(range(0, na, every)) | {i % na for i in (-2, -1, 1, 2, na // 2 - 1, na // 2, na // 2 + 1)})
    admitted, outside, reversed_ = _batches(nx, ny, na, nb, pixel_mm, bin_mm, views, (8, 16, 32))
    assert outside == 0 and reversed_ == 0
    if min(nx, ny) >= 29:
        assert admitted > 0


def test_a_band_moves_the_point_by_many_ulps():
    worst = math.inf
    for na in range(1, 1025):
        for i in range(na):
            _, cm, cn = _slope(i, na)
            if cn == 0.0:
                continue                         # the points of a ray along the axis are all the same
            du = abs(cn / cm)
            largest = 0.5 + 8192.0 * du          # |uf| <= 0.5 and at most 8192 bands from the centre
            worst = min(worst, du / float(np.spacing(f32(largest))))
    assert worst > 8.0                           # the three roundings of two neighbours: 3 ulps at most
