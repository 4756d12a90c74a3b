"""The solver's projectors on either side of their choice between parts of a
ray per warp (small detectors) and a thread per ray: detectors of one and a few
pixels, ragged ones, and one past the line, against the FP64 oracle (J 1e-4,
dJ/dw 1e-3, the tolerances of the other parity tests), and with empty-space
skipping on and off, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1102_1712_gb300 import synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1102_1712_gb300 import build as B
    B.build()
    from paper_1102_1712_gb300 import pcasolve
    return pcasolve


def problem(det, angle):
    vol = S.volume(45, 39, 20, 4.0, 4.0, 4.0)
    f0, _ = S.phantom(vol, 10.0, seed=21)
    f0 = (f0 * (1 + 0.05 * S.rng(22).uniform(-1, 1, f0.shape))).astype(np.float32)
    U = S.eigen_dvfs(vol, 2, seed=23)
    cb = S.cone_beam(det[0], det[1], 220.0 / max(det[0], 4), 130.0 / max(det[1], 4), angle)
    y = O.drr_forward(O.warp_volume(f0, O.pca_dvf(None, U, np.array([0.9, -0.3]), vol), vol), vol, cb, 2.0)
    y = (y / 1.2 - 0.1 + S.gaussian_noise(y.shape, 0.01 * y.max(), seed=24, dtype=np.float64)).astype(np.float32)
    d = [torch.from_numpy(np.ascontiguousarray(t).ravel()).cuda() for t in (f0, U, y)]
    return vol, cb, f0, U, y, d


@pytest.mark.parametrize("angle", [0.4, 1.6])
@pytest.mark.parametrize("det", [(3, 2), (1, 40), (33, 17), (161, 121), (403, 391)])
def test_split_projectors(P, det, angle):
    vol, cb, f0, U, y, (df0, dU, dy) = problem(det, angle)
    w = np.array([0.5, 0.1])
    J, G, ab = P.cost_grad(df0, None, dU, w, dy, vol, cb, 2.0)
    Jr, Gr, abr = O.cost_grad(f0, None, U, w, y, vol, cb, 2.0)
    assert abs(J - Jr) <= 1e-4 * Jr and np.linalg.norm(G - Gr) <= 1e-3 * np.linalg.norm(Gr)
    prm = P.default_params(2.0, max_iter=3, mu_min=0.025)
    t = P.tuning_get(vol, cb, 2)
    try:
        got = []
        for skip in (1, 0):
            P.tuning_set(vol, cb, 2, dict(t, skip_empty=skip))
            got.append(P.solve_projection(df0, None, dU, dy, vol, cb, np.zeros(2), prm))
    finally:
        P.tuning_clear()
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
    wo, sto, _ = O.solve_projection(f0, None, U, y, vol, cb, np.zeros(2), prm)
    assert got[0][1]["iters"] == sto["iters"] and got[0][1]["evals"] == sto["evals"]
    assert np.abs(got[0][0] - wo).max() <= 2e-3
