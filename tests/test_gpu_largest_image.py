"""The largest image the library takes, 8192 x 8192, with as many views: its tables have
2^31 tile-view pairs.  One iteration runs from its tables, changes exactly the pixels
that the (table-free) back-projection says a ray meets, and leaves every value finite."""
import numpy as np
import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_largest_image_steps():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Reconstructor, _lib
    g = inputs.make_geometry(8192, 0.02, 8192, 1, bin_mm=1.0)
    R = Reconstructor(g, inputs.make_spectra(1, 1e5), 1e-7)
    R.set_counts(torch.full((g.n_rays, 4), 5e4, device="cuda"))
    R.step(1)
    assert _lib.osscir_memory(R.handle)[1] > 0
    met = R.backproject(torch.ones((g.n_rays, 4), device="cuda"))[:, 0] > 0
    x = R.maps()
    assert bool(torch.isfinite(x).all()) and np.isfinite(R.dtpl(1))
    assert bool((x[met][:, :3] != 0).any(1).all()) and not bool(x[~met].any())
    assert 0 < int(met.sum()) < met.numel()
    R.close()
