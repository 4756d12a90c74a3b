"""A workspace's earlier contents do not matter: every call gives the same bits
from memory full of NaN as from zeros, in both layouts of the solver volumes,
at row lengths of every alignment, with and without empty-space skipping."""
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


@pytest.mark.parametrize("skip", [1, 0])
@pytest.mark.parametrize("angle", [0.1, np.pi / 2])
@pytest.mark.parametrize("dims", [(33, 30, 9), (34, 31, 8), (35, 32, 1), (36, 29, 17)])
def test_dirty_workspace(P, dims, angle, skip):
    vol, cb = S.volume(*dims, 4.0, 4.0, 4.0), S.cone_beam(40, 25, 5.0, 5.0, angle)
    g = S.rng(3)
    f0 = g.uniform(0.0, 0.03, np.prod(dims)).astype(np.float32)
    f0[g.uniform(size=f0.size) < 0.3] = 0.0
    U = S.eigen_dvfs(vol, 2, seed=4)
    d0, dU = torch.from_numpy(f0).cuda(), torch.from_numpy(U.ravel()).cuda()
    y = P.drr_forward(d0, vol, cb, 2.0) + 0.01 * torch.from_numpy(g.standard_normal(1000).astype(np.float32)).cuda()
    w = np.array([0.4, -0.2])
    prm = P.default_params(2.0, max_iter=2, mu_min=0.025)
    got = []
    t = P.tuning_get(vol, cb, 2)
    try:
        P.tuning_set(vol, cb, 2, dict(t, skip_empty=skip))
        for fill in (0, 255):
            ws, wf = P.Workspace(vol, cb, 2), P.WorkspaceF0(vol, cb, 2)
            r = []
            for b in (ws, wf):
                b.buf.fill_(fill)
            J, G, ab = P.cost_grad(d0, None, dU, w, y, vol, cb, 2.0, ws=ws)
            r += [J, *G, *ab]
            J, _, ab, _ = P.cost_grad_f0(d0, None, dU, w, y, vol, cb, 2.0, want_grad=False, want_grad_f0=False, ws=wf)
            r += [J, *ab]
            wf.buf.fill_(fill)
            J, G, ab, df = P.cost_grad_f0(d0, None, dU, w, y, vol, cb, 2.0, ws=wf)
            r += [J, *G, *ab, *df.cpu().numpy()]
            ws.buf.fill_(fill)
            wo, st = P.solve_projection(d0, None, dU, y, vol, cb, np.zeros(2), prm, ws=ws)
            r += [*wo, st["J"], st["iters"], st["evals"]]
            got.append(np.array(r))
    finally:
        P.tuning_clear()
    assert np.isfinite(got[0]).all() and np.array_equal(got[0], got[1])
