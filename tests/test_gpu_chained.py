"""Iterations enqueued together (chained launches, csrc/capi.cu) against the same ones
enqueued one by one (each the recorded graph): state and D_TPL bit for bit, single-loop
and nested, from any phase."""
import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,views,bins,inner", [(64, 128, 128, 1), (33, 45, 61, 1), (150, 140, 170, 1), (40, 50, 60, 3)])
def test_together_equals_one_by_one(n, views, bins, inner):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Reconstructor
    g = inputs.make_geometry(n, 0.5, views, bins)
    sp = inputs.make_spectra(bins, 1e5)
    gen = torch.Generator(device="cuda").manual_seed(n)
    f = torch.rand((n * n, 4), device="cuda", generator=gen) * torch.tensor([1.0, 0.1, 0.01, 0.0], device="cuda")
    got = []
    for runs in ((1, 7, 5, 2), (1,) * 15):
        R = Reconstructor(g, sp, inputs.step_ratio(n, 1e5), inner=inner)
        R.set_counts(R.simulate(f).round())
        for k in runs:
            R.step(k)
        got.append((*R.get_state()[:3], R.dtpl(1)))
        R.close()
    for other in got[1:]:
        for a, b in zip(got[0][:3], other[:3]):
            assert torch.equal(a, b)
        assert got[0][3] == other[3]
