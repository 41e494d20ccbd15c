"""The FP32 form of the Poisson draws (csrc/noise.cu, poisson_fast) gives the FP64
definition's counts, one for one, at the edges of its ranges: the change from
inversion to rejection at a mean of 10, small means, counts near 2^24 (where it
hands over to FP64) and means at which the log test decides often."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("means", [
    (0.0, -1.0, 1e-30, 1e-6, 0.5, 3.0, 9.9999990463),
    (10.0, 10.0000009537, 11.0, 14.0, 18.5, 25.0),
    (100.0, 4096.0, 65535.5, 1.0e6, 8388607.5),
    (16777215.0, 16777216.0, 2.0e7, 3.0e7),
], ids=["inversion", "small", "large", "hand-over"])
def test_counts_equal_oracle_at_the_edges(orc, means):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import _lib
    lam = np.repeat(np.array(means, dtype=np.float32), 20_000)
    got = _lib.osscir_poisson_noise(torch.tensor(lam, device="cuda"), 99).cpu().double().numpy()
    want = orc.poisson_noise(lam.astype(np.float64), 99).astype(np.float32).astype(np.float64)
    assert np.array_equal(got, want)
    nan = _lib.osscir_poisson_noise(torch.full((33,), float("nan"), device="cuda"), 1)
    assert not nan.any()
