"""The forward table's line sums (csrc/mocca.cu, k_fp_proj) ray by ray: with zero curvature
(model 1) one iteration leaves each ray's residual c - c^ in its dual, and c^ at the same
point comes from osscir_simulate, which traces the rays.  Equal line sums give equal
exponentials; the two sums over 101 energies differ by at most 16 roundings (the plain
partial of 16 energies) and a few of products, together 2e-6 of c^.  Sizes on both sides
of the rule that picks four or eight units a trip, and rays of a few pixels to many
units."""
import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,views,bins", [
    (64, 1024, 130), (5, 1024, 130), (7, 30, 33), (130, 40, 70), (200, 380, 256), (200, 381, 256), (33, 45, 512)])
def test_every_ray(n, views, bins):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Reconstructor, osscir_footprint_rays
    g = inputs.make_geometry(n, 0.5, views, bins, start_deg=3.0)
    R = Reconstructor(g, inputs.make_spectra(bins, 1e5), inputs.step_ratio(n, 1e5), model=1)
    gen = torch.Generator(device="cuda").manual_seed(n)
    c = (torch.rand((g.n_rays, 4), device="cuda", generator=gen) * 1e4).round()
    x = torch.rand((n * n, 4), device="cuda", generator=gen) * torch.tensor([1.0, 0.2, 0.01, 0.0], device="cuda")
    R.set_counts(c)
    R.set_state(x, x, R.window_rays(), 0)
    R.step(1)
    y = R.get_state()[2].double()
    chat = R.simulate(x).double()
    cnt = torch.zeros(g.n_rays, dtype=torch.int32, device="cuda")
    osscir_footprint_rays(R.handle, 0, g.n_rays, 0, cnt, cnt, cnt)
    R.close()
    met = cnt > 0
    r = c.double() - chat
    assert bool(met.any()) and not bool(y[~met].any())
    assert bool(((y - r).abs() <= 2e-6 * chat + 2.0 ** -23 * r.abs())[met].all())
