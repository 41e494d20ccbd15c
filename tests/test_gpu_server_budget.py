"""The server's memory budget where a context's footprint tables are larger than the
estimate it is admitted by (a detector of few bins): the contexts' true sizes stay within
the budget, requests wait for one another, and one alone is served all the same."""
import time

import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _counts(g, sp):
    from paper_1801_06263_gb300 import Reconstructor
    R = Reconstructor(g, sp, 1e-7)
    f = torch.zeros((g.n_pixels, 4), device="cuda")
    f[:, :3] = torch.tensor(inputs.disk_phantom(g, radius_mm=0.2 * g.n, insert_mm=0.03 * g.n), device="cuda")
    c = R.simulate(f).round().cpu().numpy()
    R.close()
    return c


@pytest.mark.parametrize("share,peak", [(1.9, 1), (0.9, 1), (2.1, 2)])
def test_budget_holds_true_sizes(share, peak):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import _lib as L
    g = inputs.make_geometry(64, 0.5, 512, 64)
    sp = inputs.make_spectra(64, 1e5)
    c, lam = _counts(g, sp), inputs.step_ratio(64, 1e5)
    probe = L.osscir_server_create(8 << 30, 1)
    assert L.osscir_poll(probe, L.osscir_submit(probe, g, sp.s, sp.N, sp.mu, lam, c, 1), -1)[0] == 0
    size = L.osscir_server_info(probe)[2]
    L.osscir_server_destroy(probe)
    budget = int(share * size)
    srv = L.osscir_server_create(budget, 4)
    try:
        ts = [L.osscir_submit(srv, g, sp.s, sp.N, sp.mu, lam * k, c, 3000) for k in (1.0, 0.9, 0.8)]
        most = 0
        for _ in range(20000):
            r, q, b = L.osscir_server_info(srv)
            most = max(most, r)
            assert b <= max(budget, size)
            if r == 0 and q == 0:
                break
            time.sleep(0.0005)
        for t in ts:
            assert L.osscir_poll(srv, t, -1)[0] == 0
        assert most == peak
    finally:
        L.osscir_server_destroy(srv)
