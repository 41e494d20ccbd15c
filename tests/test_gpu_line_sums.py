"""The on-the-fly line sums (csrc/mocca.cu, ray_line_sum) where their two-slab trips and
three-cell slabs can go wrong: odd and tiny images, rays at 45 degrees and along the
axes, a fan that passes mostly outside.  Against the FP64 oracle at the projector tests'
2e-6 of the largest sum (FP32 weights telescope along a ray)."""
import numpy as np
import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,views,bins,start,arc", [
    (1, 8, 9, 0.0, 360.0), (2, 16, 33, 45.0, 360.0), (3, 9, 17, 0.0, 180.0), (33, 40, 65, 44.9, 0.3),
    (64, 24, 65, 0.0, 360.0), (129, 12, 200, 45.0, 90.0)])
def test_line_sums_match_oracle(orc, n, views, bins, start, arc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Reconstructor
    g = inputs.make_geometry(n, 0.5, views, bins, start_deg=start, arc_deg=arc)
    R = Reconstructor(g, inputs.make_spectra(bins, 1e5), 1e-7)
    f = np.random.default_rng(n).uniform(0.0, 1.0, (n * n, 4)).astype(np.float32)
    got = R.forward(torch.tensor(f, device="cuda")).cpu().double().numpy()
    R.close()
    want = orc.forward(g, f.astype(np.float64))
    assert np.abs(got - want).max() <= 2e-6 * np.abs(want).max()
