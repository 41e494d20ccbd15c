"""The pixel step on a box (csrc/mocca.cu, box_step3) against the oracle's active-set
enumeration, for random positive definite P up to condition 1e6 and steps that leave the
box through any face, edge or corner.  Tolerance: the double-float solve is within
2^-44 cond = 6e-8 of the step, the FP32 result within 6e-8 of its size; 1e-6 of
both together leaves a factor of ten.  Steps that stay in the box are the free step's
(its double-float adjugate has an error of its own on such matrices) and are not part
of this."""
import numpy as np
import pytest

from paper_1801_06263_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
INF = float("inf")


@pytest.mark.parametrize("lo,hi", [
    ((0.0, 0.0, 0.0), (INF, INF, INF)),
    ((-0.25, 0.0, 0.1), (1.0, 0.5, 0.2)),
    ((-INF, 0.0, 0.3), (0.5, INF, 0.3)),
    ((-INF, -INF, -INF), (0.25, INF, 0.0)),
], ids=["nonnegative", "box", "half-open and equal", "upper"])
def test_box_step_matches_oracle(orc, lo, hi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_06263_gb300 import Reconstructor, _lib
    g = inputs.make_geometry(64, 0.5, 4, 64)
    lam, P = float(np.float32(1e-3)), 64 * 64
    rng = np.random.default_rng(3)
    Q = np.linalg.qr(rng.normal(size=(P, 3, 3)))[0]
    w = 10.0 ** rng.uniform(-6.0, 0.0, (P, 3))
    M = np.einsum("pij,pj,pkj->pik", Q, w, Q).astype(np.float32)
    x = rng.uniform(-0.1, 0.6, (P, 3)).astype(np.float32)
    step = rng.normal(size=(P, 3)) * 10.0 ** rng.uniform(-2.0, 0.5, (P, 1))
    v = np.einsum("pij,pj->pi", M.astype(np.float64) / lam, step).astype(np.float32)
    R = Reconstructor(g, inputs.make_spectra(64, 1e4), lam, box=(lo, hi))
    x4 = torch.zeros((P, 4), device="cuda")
    x4[:, :3] = torch.tensor(x)
    R.set_state(x4, x4, R.window_rays(), 0)
    chan = torch.tensor(np.concatenate([v.T, M[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]].T]), device="cuda").contiguous()
    _lib.osscir_mocca_apply(R.handle, chan)
    got = R.maps().cpu().double().numpy()[:, :3]
    R.close()
    lo32, hi32 = np.float32(lo).astype(np.float64), np.float32(hi).astype(np.float64)
    worst, outside = 0.0, 0
    for k in range(P):
        T = M[k].astype(np.float64) / lam
        T = np.triu(T) + np.triu(T, 1).T
        free = x[k].astype(np.float64) - np.linalg.solve(T, v[k].astype(np.float64))
        if (free >= lo32).all() and (free <= hi32).all():
            continue
        want = orc.primal_update(T, v[k].astype(np.float64), x[k].astype(np.float64), box=(lo32, hi32))
        size = np.abs(x[k]).max() + np.abs(np.linalg.solve(T, v[k])).max() + np.abs(want).max()
        outside += 1
        worst = max(worst, np.abs(got[k] - want).max() / size)
    assert worst < 1e-6 and outside > P // 4, (worst, outside)
    assert (got >= lo32 - 0.0).all() and (got <= hi32 + 0.0).all()
