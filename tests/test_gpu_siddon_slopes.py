"""drr_siddon on rays nearly parallel to a voxel plane, against the exact path.
The central detector column of an odd detector looks through the isocentre,
where an even number of voxels along x has a face: with one value on each side
of that face the path is half the chord times either, whatever the slope m
(voxels of x per layer of y).  Only the crossing of the face can go wrong, by
what the position along x is wrong, over m, in layers:
  position: 8 roundings of doubles no larger than nx, and per layer the rounding
  of the 48-bit slope (2^-49 voxel), the entry's another;
  crossing: float's 2^-24 of a layer twice;
and the result is rounded to float (2^-24), its scale in double."""
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


ANGLES = [1e-9, -1e-8, 1e-7, float(np.float32(np.pi)), 1e-6, -3e-5, 1e-3, 0.0039, 0.00391, 0.01, -0.06, 0.2]


@pytest.mark.parametrize("angle", ANGLES)
@pytest.mark.parametrize("nx,ny", [(64, 61), (64, 62), (190, 223)])
def test_face_through_the_isocentre(P, angle, nx, ny):
    nz, s = 8, 2.0
    vol = S.volume(nx, ny, nz, s, s, s)
    lo, hi = np.float32(0.01), np.float32(0.03)
    f = np.full((nz, ny, nx), hi, np.float32)
    f[:, :, :nx // 2] = lo
    cb = S.cone_beam(33, 8, 4.0, 1.0, angle)
    p = P.drr_siddon(torch.from_numpy(f.ravel()).cuda(), vol, cb).cpu().numpy().reshape(8, 33)[:, 16]
    v = (np.arange(8) - 3.5) * 1.0
    chord = ny * s / abs(np.cos(angle)) * np.sqrt(1.0 + (v / cb["sdd"]) ** 2)          # enters and leaves by y faces
    m = abs(np.tan(angle))
    exact = 0.5 * (float(lo) + float(hi)) * chord
    position = 8 * 2.0 ** -53 * nx + 2.0 ** -49 * (ny + 1)
    tol = 2.0 ** -23 * exact + (position / m + 2.0 ** -23) * float(hi - lo) * chord / ny
    assert (np.abs(p - exact) <= tol).all(), np.abs(p - exact) / tol
