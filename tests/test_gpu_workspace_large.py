"""A workspace's earlier contents do not matter on a detector past the sizes of
the split projectors either (a thread per ray: through L1 and staged), in both
layouts: the same bits from memory full of NaN as from zeros."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("chunk1", [0, 32])
@pytest.mark.parametrize("angle", [0.1, np.pi / 2])
@pytest.mark.parametrize("dims", [(33, 30, 9), (36, 29, 17)])
def test_dirty_workspace(P, dims, angle, chunk1):
    vol, cb = S.volume(*dims, 4.0, 4.0, 4.0), S.cone_beam(403, 391, 0.5, 0.4, angle)
    g = S.rng(3)
    f0 = g.uniform(0.0, 0.03, np.prod(dims)).astype(np.float32)
    f0[g.uniform(size=f0.size) < 0.3] = 0.0
    U = S.eigen_dvfs(vol, 2, seed=4)
    d0, dU = torch.from_numpy(f0).cuda(), torch.from_numpy(U.ravel()).cuda()
    noise = torch.from_numpy(g.standard_normal(403 * 391).astype(np.float32)).cuda()
    y = P.drr_forward(d0, vol, cb, 2.0) + 0.01 * noise
    w = np.array([0.4, -0.2])
    got = []
    t = P.tuning_get(vol, cb, 2)
    try:
        P.tuning_set(vol, cb, 2, dict(t, chunk1=chunk1))
        for fill in (0, 255):
            ws = P.Workspace(vol, cb, 2)
            ws.buf.fill_(fill)
            J, G, ab = P.cost_grad(d0, None, dU, w, y, vol, cb, 2.0, ws=ws)
            ws.buf.fill_(fill)
            wo, st = P.solve_projection(d0, None, dU, y, vol, cb, np.zeros(2),
                                        P.default_params(2.0, max_iter=2, mu_min=0.025), ws=ws)
            got.append(np.array([J, *G, *ab, *wo, st["J"], st["iters"], st["evals"]]))
    finally:
        P.tuning_clear()
    assert np.isfinite(got[0]).all() and np.array_equal(got[0], got[1])
