"""The back-projection table for fine detectors (csrc/mocca.cu): 16-bit stage slots (a step
between slots that a signed byte cannot hold), the larger stage where a tile's bins in one
view exceed kBTSlots = 396, and no table where they exceed kBTSlotsFine = 564.  Two
iterations against the FP64 oracle and split view ranges against the whole, at the
tolerances of test_gpu_bp_table.py (a pixel adds fewer terms here than there); a batch
that mixes stage sizes against the single solves, bit for bit."""
import numpy as np
import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(n, views, bins):
    g = inputs.make_geometry(n, 0.5, views, bins, start_deg=3.0)
    sp = inputs.make_spectra(bins, 1e5)
    f = np.zeros((n * n, 3))
    f[:, 0] = 1.0
    f[:, 2] = 0.002 * (np.arange(n * n) % 3)
    return g, sp, f, inputs.step_ratio(n, 1e5)


def _largest_step(g):
    """The largest step from a tile's first bin to a pixel's first bin in view 0, whose
    rays open a chunk: exact shadows of the first tile and of its pixels."""
    th = np.deg2rad(g.start_deg)
    c, s = np.cos(th), np.sin(th)
    m = min(16, g.n)
    i = -0.5 * g.n * g.pixel_mm + g.pixel_mm * np.arange(m + 1)
    X, Y = i[None, :], i[:, None]
    beta = g.sdd_mm / g.bin_mm * (c * Y - s * X) / (g.sid_mm - (c * X + s * Y)) + 0.5 * (g.n_bins - 1)
    low = np.minimum(np.minimum(beta[:-1, :-1], beta[1:, :-1]), np.minimum(beta[:-1, 1:], beta[1:, 1:]))
    first = np.maximum(0, np.ceil(low))
    return first.max() - first.min()


def _forward_table_bytes(R, g):
    """Table bytes without the back-projection's part (osscir_launch.h, FpTables)."""
    from paper_1801_06263_gb300 import osscir_footprint_rays
    groups = (g.n_bins + 31) // 32
    cnt = torch.zeros(g.n_rays, dtype=torch.int32, device="cuda")
    osscir_footprint_rays(R.handle, 0, g.n_rays, 0, cnt, cnt, cnt)
    unit = torch.zeros((g.n_views, groups * 32), dtype=torch.int64, device="cuda")
    unit[:, :g.n_bins] = (cnt.view(g.n_views, g.n_bins) + 3) // 4
    units = int(unit.view(g.n_views, groups, 32).amax(2).sum())
    spans = ((g.n + 15) // 16) ** 2 * g.n_views
    return (units + 1) * 768 + 8 * g.n_rays + 4 * (g.n_views * groups + 1) + 4 * spans


@pytest.mark.parametrize("n,views,bins,table,wide", [
    (33, 45, 512, True, True), (32, 40, 896, True, True), (64, 21, 2048, True, True), (8, 30, 512, True, True),
    (1, 30, 560, True, False), (8, 20, 1500, False, False)])
def test_fine_detector(orc, n, views, bins, table, wide):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Reconstructor, _lib
    g, sp, f, lam = _problem(n, views, bins)
    if wide:
        assert _largest_step(g) >= 130
    sp32 = inputs.Spectra(sp.energies, sp.s.astype(np.float32).astype(np.float64),
                          sp.N.astype(np.float32).astype(np.float64), sp.mu.astype(np.float32).astype(np.float64))
    c = np.random.default_rng(n).poisson(orc.counts(g, sp32, f)).astype(np.float32)
    R = Reconstructor(g, sp, lam)
    R.set_counts(torch.tensor(c, device="cuda"))
    R.step(2)
    assert (_lib.osscir_memory(R.handle)[1] > _forward_table_bytes(R, g)) == table
    got = R.maps().cpu().double().numpy()[:, :3]
    st, _ = orc.mocca(g, sp32, c.astype(np.float64), 2, float(np.float32(lam)))
    assert np.linalg.norm(got - st.x) <= 1e-5 * np.linalg.norm(st.x)
    state = R.get_state()
    whole = torch.zeros((9, n * n), device="cuda")
    _lib.osscir_mocca_partial(R.handle, 0, views, whole)
    total = torch.zeros_like(whole)
    cut = [0, 1, views // 3, views - 1, views]
    for v0, v1 in zip(cut, cut[1:]):
        R.set_state(*state)
        part = torch.zeros_like(whole)
        _lib.osscir_mocca_partial(R.handle, v0, v1, part)
        total += part
    R.close()
    for ch in range(9):
        assert (total[ch] - whole[ch]).norm() <= 1e-6 * whole[ch].norm() + 1e-6 * whole.abs().max()


def test_batch_of_stage_sizes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Batch, Reconstructor
    plain, together = [], []
    for out in (plain, together):
        for n, views, bins in ((32, 40, 896), (64, 40, 64), (33, 45, 512)):
            g, sp, f, lam = _problem(n, views, bins)
            R = Reconstructor(g, sp, lam)
            f4 = torch.zeros((n * n, 4), device="cuda")
            f4[:, :3] = torch.tensor(f, dtype=torch.float32)
            R.set_counts(R.simulate(f4).round())
            out.append(R)
    for R in plain:
        R.step(3)
    for autotune in (False, True):
        for R in together:
            R.set_state(R.image(), R.image(), R.window_rays(), 0)
        B = Batch(together, autotune=autotune)
        B.step(3)
        for a, b in zip(plain, together):
            for u, v in zip(a.get_state()[:3], b.get_state()[:3]):
                assert torch.equal(u, v)
        B.close()
    for R in plain + together:
        R.close()
