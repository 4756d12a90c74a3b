"""Voxels much taller across than along z, where backprojections gather per voxel
instead of walking columns: P^T, dJ/dw and dJ/df0 against the FP64 oracle on both
sides of that line (1e-4 of the maximum, dJ/dw 1e-3, as in the other tests), and
the time of P^T on 16x16x96 voxels of 20 x 20 x 1.25 mm against 20 x 20 x 4 mm at
half a voxel a step.  The samples near a voxel are as many, so a gather takes about
the same time for both (0.77 to 1.0); walking columns took 3.5 times as long."""
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


@pytest.mark.parametrize("off_v", [0.0, 5.0])
@pytest.mark.parametrize("dims,s", [((9, 7, 33), (20.0, 18.0, 1.0)), ((9, 7, 33), (20.0, 18.0, 6.0)),
                                    ((41, 38, 150), (4.0, 4.0, 0.5)), ((41, 38, 30), (4.0, 4.0, 4.0))])
def test_against_the_oracle(P, dims, s, off_v):
    vol, cb = S.volume(*dims, *s), S.cone_beam(40, 31, 6.0, 5.0, 0.8, off_u=4.0, off_v=off_v)
    g, step = S.rng(6), 0.5 * min(s)
    img = g.uniform(0.5, 1.5, 1240).astype(np.float32)
    got = P.drr_adjoint(torch.from_numpy(img).cuda(), vol, cb, step).cpu().numpy()
    ref = O.drr_adjoint(img.reshape(31, 40).astype(np.float64), vol, cb, step).ravel()
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()
    f0, _ = S.phantom(vol, 12.0, seed=7)
    f0 = (f0 * g.uniform(0.9, 1.1, f0.shape)).astype(np.float32).ravel()
    U = S.eigen_dvfs(vol, 2, seed=8)
    w = np.array([0.4, -0.3])
    dU, d0, y = torch.from_numpy(U.ravel()).cuda(), torch.from_numpy(f0).cuda(), torch.from_numpy(img).cuda()
    J, G, _, df = P.cost_grad_f0(d0, None, dU, w, y, vol, cb, step)
    Jo, Go, _ = O.cost_grad(f0, None, U, w, img.astype(np.float64), vol, cb, step)
    _, fo, _ = O.cost_grad_f0(f0, None, U, w, img.astype(np.float64), vol, cb, step)
    assert abs(J - Jo) <= 1e-4 * Jo and np.linalg.norm(G - Go) <= 1e-3 * np.linalg.norm(Go)
    assert np.abs(df.cpu().numpy() - fo).max() <= 1e-4 * np.abs(fo).max()


def test_time_of_flat_voxels(P):
    img = torch.rand(300 * 225, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    out = torch.empty(16 * 16 * 96, device="cuda")

    def ms(sz):
        vol = P.vol_struct(S.volume(16, 16, 96, 20.0, 20.0, sz))
        cb = P.cb_struct(S.cone_beam(300, 225, 1.3, 1.3, 0.9))
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(4):
            P.drr_adjoint(img, vol, cb, 0.5 * sz, out=out)
        b.record()
        b.synchronize()
        return a.elapsed_time(b)

    t = np.min([[ms(1.25), ms(4.0)] for _ in range(8)][2:], axis=0)
    assert t[0] <= 1.5 * t[1], t
