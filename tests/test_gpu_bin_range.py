"""The pixel-driven kernels' candidate bins (csrc/osscir_internal.cuh, box_bin_range) where
rounding is largest: the pixels' footprints hold as many rays as the rays' footprints
hold pixels for fine detectors and a source just outside the image, and the projectors
give the same bits whatever the unit of length (a power of two scales every FP32 and
FP64 operation of theirs exactly)."""
import math

import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _context(n, pixel, views, bins, sid, sdd, start=13.0, arc=360.0, unit=1.0):
    from paper_1801_06263_gb300 import Reconstructor
    reach = sdd * math.tan(math.asin(min(0.999, n * pixel / math.sqrt(2.0) / sid)))
    g = inputs.Geometry(n, pixel * unit, views, bins, 2.02 * reach / bins * unit, sid * unit, sdd * unit, arc, start)
    return Reconstructor(g, inputs.make_spectra(bins, 1e5), 1e-7)


@pytest.mark.parametrize("n,pixel,views,bins,sid,sdd,start,arc", [
    (512, 0.5, 2, 8192, 181.1, 400.0, 44.5, 180.0), (700, 0.05, 3, 30000, 25.0, 300.0, 37.5, 45.0),
    (64, 0.5, 9, 2048, 500.0, 1000.0, 13.0, 360.0)])
def test_pixel_footprints_hold_every_ray(n, pixel, views, bins, sid, sdd, start, arc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import osscir_footprint_pixels, osscir_footprint_rays
    R = _context(n, pixel, views, bins, sid, sdd, start, arc)
    L, P, cap = views * bins, n * n, 2 * n + 4
    cnt = torch.zeros(L, dtype=torch.int32, device="cuda")
    idx = torch.zeros((L, cap), dtype=torch.int32, device="cuda")
    wt = torch.zeros((L, cap), dtype=torch.float32, device="cuda")
    osscir_footprint_rays(R.handle, 0, L, cap, cnt, idx, wt)
    assert int(cnt.max()) <= cap
    met = idx[torch.arange(cap, device="cuda")[None, :] < cnt[:, None]].long()
    pix = torch.zeros(P, dtype=torch.int32, device="cuda")
    osscir_footprint_pixels(R.handle, 0, P, 0, pix, idx, wt)
    assert torch.equal(torch.bincount(met, minlength=P), pix.long())
    R.close()


@pytest.mark.parametrize("unit", [2.0 ** 70, 2.0 ** -60])
def test_projectors_in_any_unit_of_length(unit):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gen = torch.Generator(device="cuda").manual_seed(7)
    x = torch.rand((50 * 50, 4), device="cuda", generator=gen)
    y = torch.rand((61 * 77, 4), device="cuda", generator=gen)
    got = []
    for u in (1.0, unit):
        R = _context(50, 0.5, 61, 77, 500.0, 1000.0, unit=u)
        got.append((R.forward(x) / u, R.backproject(y) / u))
        R.close()
    assert got[0][1].abs().max() > 0
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
