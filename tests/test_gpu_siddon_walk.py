"""The layer walk of drr_siddon against the FP64 oracle where it can go wrong:
one voxel or one plane, rays along an axis (through voxel centres and along
faces), the steepest axis being z, rays that cut a corner, layers crossed by
two faces, signs of every direction, infinite values.  Tolerance: 1e-6 of the
maximum, as in the other Siddon tests (the result is rounded once to float)."""
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


CASES = [((1, 1, 1, 40.0, 30.0, 20.0), (21, 17, 4.0, 4.0), 0.3, (0.0, 0.0)),
         ((37, 1, 9, 4.0, 60.0, 4.0), (31, 29, 6.0, 4.0), 1.9, (0.0, 0.0)),
         ((31, 33, 17, 4.0, 4.0, 4.0), (41, 31, 5.0, 4.0), 0.0, (0.0, 0.0)),       # central ray through voxel centres
         ((31, 33, 17, 4.0, 4.0, 4.0), (41, 31, 5.0, 4.0), np.pi, (1.0, 1.0)),
         ((30, 34, 16, 4.0, 4.0, 4.0), (41, 31, 5.0, 4.0), 0.0, (0.0, 0.0)),       # and along faces
         ((12, 10, 90, 20.0, 20.0, 0.5), (31, 61, 8.0, 9.0), 0.6, (0.0, 0.0)),     # steepest in z
         ((40, 40, 40, 3.0, 3.0, 3.0), (60, 60, 4.0, 4.0), 2.0, (60.0, 60.0)),     # corners
         ((53, 47, 21, 3.0, 3.0, 5.0), (64, 48, 4.0, 4.0), 3.9, (-9.0, 7.0)),
         ((53, 47, 21, 3.0, 3.0, 5.0), (64, 48, 4.0, 4.0), 5.5, (0.0, -7.0))]


@pytest.mark.parametrize("dims,det,angle,off", CASES)
def test_siddon_walk(P, dims, det, angle, off):
    vol = S.volume(*dims)
    f = S.rng(7).uniform(0.01, 0.03, dims[2] * dims[1] * dims[0]).astype(np.float32)
    cb = S.cone_beam(det[0], det[1], det[2], det[3], angle, off_u=off[0], off_v=off[1])
    p = P.drr_siddon(torch.from_numpy(f).cuda(), vol, cb).cpu().numpy().astype(np.float64)
    po = O.siddon_forward(f.astype(np.float64), vol, cb)
    assert po.max() > 0 and np.abs(p - po).max() <= 1e-6 * po.max()


def test_siddon_infinite_voxel(P):
    vol, cb = S.volume(20, 21, 9, 4.0, 4.0, 4.0), S.cone_beam(40, 30, 4.0, 4.0, 0.7)
    f = np.full((9, 21, 20), 0.02, np.float32)
    one = np.zeros_like(f)
    f[4, 9, 11], one[4, 9, 11] = np.inf, 1.0
    p = P.drr_siddon(torch.from_numpy(f.ravel()).cuda(), vol, cb).cpu().numpy()
    hit = O.siddon_forward(one, vol, cb)
    assert np.isposinf(p[hit > 1e-6]).all() and np.isfinite(p[hit == 0.0]).all()
