"""The candidate bins of a box of pixels in a view (csrc/osscir_internal.cuh, box_bin_range)
cover the box's exact shadow: the FP32 formula, restated in numpy with the fast division
2 ulp off either way, against the FP64 detector coordinates of the four corners, for the
boxes that the library asks for (a pixel, two pixels one above the other, a 16 x 16 tile,
tiles and pairs cut by the image's edge).  Detectors from coarse to as fine as the tables
take, sources from far away to just outside the image, lengths in units from 2^-60 to
2^70 mm."""
import numpy as np
import pytest

from paper_1801_06263_gb300 import inputs

F = np.float32


def _fma(a, b, c):   # the product of two FP32 values is exact in FP64
    return np.asarray(np.float64(a) * np.float64(b) + np.float64(c)).astype(F)


def _range32(g, c, s, X, Y, hx, hy, off):
    """box_bin_range; off: the relative error of both divisions."""
    c, s, R = F(c), F(s), g.n * g.pixel_mm / np.sqrt(2.0)
    sid, scale, mid = F(g.sid_mm), F(g.sdd_mm / g.bin_mm), F(0.5 * (g.n_bins - 1))
    slack_num, slack_den = F(48 * 2.0 ** -24 * R), F(48 * 2.0 ** -24 * g.sid_mm)
    num, den = _fma(c, Y, -s * X), sid - _fma(c, X, s * Y)
    den_min = np.maximum(den - _fma(hx, abs(c), _fma(hy, abs(s), slack_den)), F(1e-6) * den)
    r = (num / den) * F(1 + off)
    reach = _fma(hx, abs(_fma(c, r, -s)), _fma(hy, abs(_fma(s, r, c)), _fma(slack_den, abs(r), slack_num)))
    beta = _fma(scale, r, mid)
    half = _fma(scale, (reach / den_min) * F(1 - off), F(0.01 + 2.0 ** -22 * g.n_bins))
    lo = np.maximum(0, -np.floor(np.clip(half - beta, F(-1e9), F(1e9))))
    return lo, np.minimum(g.n_bins - 1, np.floor(np.clip(beta + half, F(-1e9), F(1e9))))


@pytest.mark.parametrize("w,h", [(1, 1), (1, 2), (16, 16)])
@pytest.mark.parametrize("n,pixel,bins,sid,sdd,cover,unit", [
    (256, 0.5, 512, 500.0, 1000.0, 1.0, 1.0), (37, 0.7, 300, 18.4, 60.0, 0.5, 1.0), (64, 0.5, 64, 1e6, 1.001e6, 1.0, 1.0),
    (4096, 0.05, 65535, 500.0, 1000.0, 1.0, 1.0), (2700, 0.05, 65535, 100.0, 1000.0, 1.0, 1.0),
    (512, 0.5, 8192, 181.1, 400.0, 1.0, 1.0), (2048, 0.1, 50000, 145.0, 300.0, 1.0, 1.0),
    (50, 0.5, 77, 500.0, 1000.0, 1.0, 2.0 ** 70), (50, 0.5, 77, 500.0, 1000.0, 1.0, 2.0 ** -60)])
def test_candidate_bins_cover_the_box(n, pixel, bins, sid, sdd, cover, unit, w, h):
    reach = sdd * np.tan(np.arcsin(min(0.999, n * pixel / np.sqrt(2.0) / sid)))   # of the image on the detector
    g = inputs.Geometry(n, pixel * unit, 1, bins, 2.02 * cover * reach / bins * unit, sid * unit, sdd * unit)
    rng = np.random.default_rng(n + w)
    ix, iy = rng.integers(0, (n + w - 1) // w, 40000) * w, rng.integers(0, (n + h - 1) // h, 40000) * h
    ix[:4000] = rng.integers(0, 3, 4000) * w      # enough of them near a corner of the image
    iy[:4000] = rng.integers(0, 3, 4000) * h
    ix, iy = np.minimum(ix, n - 1), np.minimum(iy, n - 1)
    jx, jy = np.minimum(n, ix + w), np.minimum(n, iy + h)
    x0 = -0.5 * n * g.pixel_mm
    planes = [_fma(i.astype(F), F(g.pixel_mm), F(x0)) for i in (ix, jx, iy, jy)]
    exact = [x0 + i * g.pixel_mm for i in (ix, jx, iy, jy)]
    if (w, h) == (1, 1):     # as pixel_bin_range and pair_entries form the centre and the half sides
        hx = hy = F(0.5) * F(g.pixel_mm)
        X, Y = planes[0] + hx, planes[2] + hy
    elif (w, h) == (1, 2):
        hx = F(0.5) * F(g.pixel_mm)
        two = iy + 1 < n
        hy = np.where(two, F(g.pixel_mm), hx)
        X, Y = planes[0] + hx, np.where(two, _fma((iy + 1).astype(F), F(g.pixel_mm), F(x0)), planes[2] + hx)
    else:
        X, Y = F(0.5) * (planes[0] + planes[1]), F(0.5) * (planes[2] + planes[3])
        hx, hy = F(0.5) * (planes[1] - planes[0]), F(0.5) * (planes[3] - planes[2])
    for th in np.concatenate([np.arange(16) * np.pi / 8, rng.uniform(0, 2 * np.pi, 24)]):
        c, s = np.cos(th), np.sin(th)
        beta = [g.sdd_mm / g.bin_mm * (c * Y1 - s * X1) / (g.sid_mm - (c * X1 + s * Y1)) + 0.5 * (bins - 1)
                for X1 in exact[:2] for Y1 in exact[2:]]
        first, last = np.maximum(0, np.ceil(np.min(beta, 0))), np.minimum(bins - 1, np.floor(np.max(beta, 0)))
        some = first <= last
        for off in (-2.0 ** -22, 2.0 ** -22):
            lo, hi = _range32(g, c, s, X, Y, hx, hy, off)
            assert (lo[some] <= first[some]).all() and (hi[some] >= last[some]).all()
            # and no more than a few bins wider where the box is far from the source
            if sid > 1.5 * n * pixel and w * h <= 2:
                assert (hi - lo - (last - first))[some].max() <= 4
