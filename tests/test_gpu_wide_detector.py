"""The projections of a detector with more bins than a grid's second dimension has groups
of 32 (65535): osscir_forward, osscir_simulate and osscir_dtpl take
it as any other.  The ones' line sums against the library's own chords."""
import numpy as np
import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("views,bins", [(1, 2200000)])
def test_wide_detector(views, bins):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Reconstructor, osscir_footprint_rays
    g = inputs.make_geometry(3, 0.5, views, bins)
    sp = inputs.Spectra(np.array([60.0]), np.ones((bins, 1, 4), np.float32), np.full((bins, 4), 1e4, np.float32),
                        np.array([[0.02], [0.05], [0.1]]))
    R = Reconstructor(g, sp, 1e-7)
    f = torch.ones((9, 4), device="cuda")
    got = R.forward(f)
    cnt = torch.zeros(g.n_rays, dtype=torch.int32, device="cuda")
    idx = torch.zeros((g.n_rays, 8), dtype=torch.int32, device="cuda")
    wt = torch.zeros((g.n_rays, 8), dtype=torch.float32, device="cuda")
    osscir_footprint_rays(R.handle, 0, g.n_rays, 8, cnt, idx, wt)
    assert int(cnt.max()) <= 8 and int(cnt.min()) < int(cnt.max())
    chord = (wt * (torch.arange(8, device="cuda")[None, :] < cnt[:, None])).sum(1)
    assert float((got - chord[:, None]).abs().max()) <= 1e-6 * float(chord.max())   # eight FP32 additions
    chat = R.simulate(f)
    want = 1e4 * torch.exp(-0.17 * chord.double())[:, None]
    assert float((chat.double() / want - 1).abs().max()) <= 1e-5
    R.set_counts(chat)
    R.set_state(f, f, R.window_rays(), 0)
    assert R.dtpl(0) <= 1e-6 * float(chat.double().sum())
    R.close()
