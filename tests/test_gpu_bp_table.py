"""The blocked back-projection table (csrc/mocca.cu) at the sizes where it can go wrong:
images that are no multiple of a tile or of a pixel pair, fewer views than view groups,
16-bit slots (a tile seen by more bins than a signed byte steps over), a chunk that ends
mid-group and view ranges that straddle chunks.  Two iterations against the FP64 oracle
(relative L2 1e-5: a few FP32 roundings of sums whose pixels the double-float step
solves), and the sums over split view ranges against the whole's (1e-6: another order
of the same FP32 additions)."""
import numpy as np
import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,views,bins", [(33, 45, 256), (16, 24, 24), (50, 61, 77), (47, 130, 64), (1, 40, 33)])
def test_table_backprojection(orc, n, views, bins):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Reconstructor, _lib
    g = inputs.make_geometry(n, 0.5, views, bins, start_deg=3.0)
    sp = inputs.make_spectra(bins, 1e5)
    sp32 = inputs.Spectra(sp.energies, sp.s.astype(np.float32).astype(np.float64),
                          sp.N.astype(np.float32).astype(np.float64), sp.mu.astype(np.float32).astype(np.float64))
    f = np.zeros((n * n, 3))
    f[:, 0] = 1.0
    f[:, 2] = 0.002 * (np.arange(n * n) % 3)
    c = np.random.default_rng(n).poisson(orc.counts(g, sp32, f)).astype(np.float32)
    lam = inputs.step_ratio(n, 1e5)
    R = Reconstructor(g, sp, lam)
    R.set_counts(torch.tensor(c, device="cuda"))
    R.step(2)
    assert _lib.osscir_memory(R.handle)[1] > 0
    got = R.maps().cpu().double().numpy()[:, :3]
    st, _ = orc.mocca(g, sp32, c.astype(np.float64), 2, float(np.float32(lam)))
    assert np.linalg.norm(got - st.x) <= 1e-5 * np.linalg.norm(st.x)
    x, xbar, y, it = R.get_state()
    whole = torch.zeros((9, n * n), device="cuda")
    _lib.osscir_mocca_partial(R.handle, 0, views, whole)
    total = torch.zeros_like(whole)
    cut = [0, 1, views // 3, views // 3 + 1, views - 1, views]
    for v0, v1 in zip(cut, cut[1:]):
        R.set_state(x, xbar, y, it)
        part = torch.zeros_like(whole)
        _lib.osscir_mocca_partial(R.handle, v0, v1, part)
        total += part
    R.close()
    for ch in range(9):
        assert (total[ch] - whole[ch]).norm() <= 1e-6 * whole[ch].norm() + 1e-6 * whole.abs().max()


@pytest.mark.parametrize("n,views,bins", [(5, 1024, 130), (64, 1024, 130), (7, 30, 33), (130, 40, 70)])
def test_table_forward_projection(n, views, bins):
    """The forward table's line sums against the on-the-fly projection's through D_TPL at one
    point, for rays of few and many units and grids that take its four-unit form (over
    912 blocks) and its eight-unit one.  Both counts are within 2e-6 of the model's, and far
    from the solution D_TPL changes by less than ten times the relative change of a count:
    1e-4 leaves a factor of five."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Reconstructor
    g = inputs.make_geometry(n, 0.5, views, bins, start_deg=3.0)
    R = Reconstructor(g, inputs.make_spectra(bins, 1e5), inputs.step_ratio(n, 1e5))
    gen = torch.Generator(device="cuda").manual_seed(n)
    R.set_counts(torch.rand((g.n_rays, 4), device="cuda", generator=gen) * 1e4)
    x = torch.rand((n * n, 4), device="cuda", generator=gen) * torch.tensor([1.0, 0.2, 0.01, 0.0], device="cuda")
    R.set_state(x, x, R.window_rays(), 0)
    fly = R.dtpl(0)
    R.step(1)
    assert abs(R.dtpl(1) - fly) <= 1e-4 * abs(fly)
    R.close()
