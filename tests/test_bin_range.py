"""The candidate bins of a pixel in a view (csrc/osscir_internal.cuh, pixel_bin_range)
cover the pixel's exact shadow: the FP32 formula, restated in numpy, against the FP64
detector coordinates of the four corners, for geometries from a distant source to one
just outside the image and from coarse to fine detector bins."""
import numpy as np
import pytest

from paper_1801_06263_gb300 import inputs

F = np.float32


def _range32(g, c, s, ix, iy):
    h, x0 = F(g.pixel_mm), F(-0.5 * g.n * g.pixel_mm)
    sid, scale, mid = F(g.sid_mm), F(g.sdd_mm / g.bin_mm), F(0.5 * (g.n_bins - 1))
    hh = F(0.5) * h
    X = (ix.astype(F) * h + x0) + hh
    Y = (iy.astype(F) * h + x0) + hh
    num = c * Y - s * X
    den = sid - (c * X + s * Y)
    den_min = np.maximum(den - hh * (abs(c) + abs(s)), F(1e-6) * den)
    reach = abs(c * num - s * den) + abs(c * den + s * num)
    beta = scale * (num / den) + mid
    half = scale * hh * (reach / (den * den_min)) + F(0.01)
    lo = np.maximum(0, -np.floor(np.clip(half - beta, -1e9, 1e9)))
    hi = np.minimum(g.n_bins - 1, np.floor(np.clip(beta + half, -1e9, 1e9)))
    return lo, hi


@pytest.mark.parametrize("n,pixel,bins,sid,sdd", [
    (256, 0.5, 512, 500.0, 1000.0), (512, 0.5, 1024, 500.0, 1000.0), (389, 0.5, 397, 500.0, 1000.0),
    (64, 0.5, 4096, 500.0, 1000.0), (37, 0.7, 61, 18.4, 60.0), (8, 3.0, 200, 17.2, 30.0), (1, 5.0, 33, 3.6, 9.0),
    (16, 0.5, 24, 5000.0, 5001.0)])
def test_candidate_bins_cover_the_shadow(n, pixel, bins, sid, sdd):
    g = inputs.make_geometry(n, pixel, 1, bins, sid_mm=sid, sdd_mm=sdd)
    iy, ix = np.divmod(np.arange(n * n), n)
    x0 = -0.5 * n * pixel
    rng = np.random.default_rng(n)
    for th in np.concatenate([np.arange(8) * np.pi / 4, rng.uniform(0, 2 * np.pi, 40)]):
        c, s = np.cos(th), np.sin(th)
        beta = []
        for a in (0, 1):
            for b in (0, 1):
                X, Y = x0 + (ix + a) * pixel, x0 + (iy + b) * pixel
                beta.append(g.sdd_mm / g.bin_mm * (c * Y - s * X) / (sid - (c * X + s * Y)) + 0.5 * (bins - 1))
        first = np.maximum(0, np.ceil(np.min(beta, 0)))
        last = np.minimum(bins - 1, np.floor(np.max(beta, 0)))
        lo, hi = _range32(g, F(c), F(s), ix, iy)
        some = first <= last
        assert (lo[some] <= first[some]).all() and (hi[some] >= last[some]).all()
