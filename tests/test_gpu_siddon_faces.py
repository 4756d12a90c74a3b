"""drr_siddon along voxel faces: where the middle of an odd detector looks along a
face between an even number of voxels (pixel coordinate and slope exactly 0), the
upper voxel's value counts, the one that a position on the face rounds down to,
over the whole chord; sizes whose half extents no double holds.  Exact: value
times chord, 2^-22 of it allowed (float's rounding of value and result)."""
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


@pytest.mark.parametrize("nv,dv", [(147, 2.3226), (31, 0.1), (95, 3.3), (11, 0.7)])
@pytest.mark.parametrize("nz,sz", [(52, 3.932), (2, 1.1), (30, 0.3)])
@pytest.mark.parametrize("angle", [0.0, 0.3, 1.0983, 2.5])
def test_row_in_a_z_face(P, nz, sz, nv, dv, angle):
    n, s = 24, 9.7
    vol, cb = S.volume(n, n, nz, s, s, sz), S.cone_beam(6, nv, 1.7, dv, angle)
    f = np.zeros((nz, n, n), np.float32)
    f[:] = (1.0 + np.arange(nz, dtype=np.float32))[:, None, None]
    p = P.drr_siddon(torch.from_numpy(f.ravel()).cuda(), vol, cb).cpu().numpy().reshape(nv, 6)[nv // 2]
    one = P.drr_siddon(torch.ones(f.size, device="cuda"), vol, cb).cpu().numpy().reshape(nv, 6)[nv // 2]
    assert (one > 0).all() and (np.abs(p - one * (1.0 + nz // 2)) <= 2.0 ** -22 * p).all()


@pytest.mark.parametrize("nu,du", [(127, 2.3226), (31, 0.1), (11, 0.7)])
@pytest.mark.parametrize("nx,sx", [(52, 3.932), (2, 1.1), (30, 0.3)])
def test_column_in_an_x_face(P, nx, sx, nu, du):
    vol, cb = S.volume(nx, 33, 9, sx, 4.3, 3.1), S.cone_beam(nu, 4, du, 1.3, 0.0)
    f = np.zeros((9, 33, nx), np.float32)
    f[:] = 1.0 + np.arange(nx, dtype=np.float32)
    p = P.drr_siddon(torch.from_numpy(f.ravel()).cuda(), vol, cb).cpu().numpy().reshape(4, nu)[:, nu // 2]
    one = P.drr_siddon(torch.ones(f.size, device="cuda"), vol, cb).cpu().numpy().reshape(4, nu)[:, nu // 2]
    assert (one > 0).all() and (np.abs(p - one * (1.0 + nx // 2)) <= 2.0 ** -22 * p).all()
