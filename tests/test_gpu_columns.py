"""The voxel-column backprojection (drr_adjoint, dJ/df0, and the gradient where
the CT has texture) against the FP64 oracle, at the shapes where it can go
wrong: one or few planes, odd and even plane counts that no chunk or tile
divides, rays along an axis, chunks of rays cut by the detector's edge, rays
over many z cells, many or few samples a voxel, with and without the mirror
symmetry in z.  Tolerances: those of the other parity tests (P^T 1e-4 of its
maximum, dJ/dw 1e-3)."""
import numpy as np
import pytest

import oracle as O
from paper_1102_1712_gb300 import synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [
    ((24, 20, 1, 4.0, 4.0, 4.0), (40, 31), (4.0, 4.0), 0.7, 0.5),        # one plane
    ((24, 20, 2, 4.0, 4.0, 4.0), (40, 31), (4.0, 4.0), 0.7, 0.5),        # the mirrored half is one plane
    ((33, 29, 17, 4.0, 4.0, 2.5), (61, 47), (3.5, 3.5), 2.4, 0.5),       # nothing divides
    ((40, 36, 33, 4.0, 3.0, 4.0), (45, 44), (5.0, 4.5), 0.0, 0.5),       # a detector column along y
    ((36, 40, 35, 3.0, 4.0, 4.0), (45, 45), (5.0, 4.5), np.pi / 2, 0.5),
    ((40, 36, 24, 4.0, 4.0, 4.0), (17, 11), (3.0, 3.0), 1.1, 0.5),       # a detector inside the volume
    ((20, 22, 41, 4.0, 4.0, 0.4), (60, 50), (2.5, 2.5), 0.3, 0.5),       # many samples a voxel, many z cells a ray
    ((30, 30, 30, 4.0, 4.0, 4.0), (50, 41), (4.5, 4.5), 0.9, 2.5),       # few samples a voxel
]
OFFSETS = [(0.0, 0.0), (6.0, -9.0)]                                      # with and without the symmetry


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1102_1712_gb300 import build as B
    B.build()
    from paper_1102_1712_gb300 import pcasolve
    return pcasolve


def view(det, pitch, angle, off):
    return S.cone_beam(det[0], det[1], pitch[0], pitch[1], angle, sad=900.0, sdd=1300.0, off_u=off[0], off_v=off[1])


@pytest.mark.parametrize("off", OFFSETS)
@pytest.mark.parametrize("dims,det,pitch,angle,ratio", SHAPES)
def test_adjoint_columns(P, dims, det, pitch, angle, ratio, off):
    vol, cb = S.volume(*dims), view(det, pitch, angle, off)
    step = ratio * min(dims[3:])
    img = S.rng(9).uniform(-1, 1, det[0] * det[1]).astype(np.float32)
    got = P.drr_adjoint(torch.from_numpy(img).cuda(), vol, cb, step).cpu().numpy().astype(np.float64)
    ref = O.drr_adjoint(img, vol, cb, step)
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()


@pytest.mark.parametrize("off", OFFSETS)
def test_nan_pixel_stays_on_its_ray(P, off):
    vol, cb = S.volume(33, 29, 17, 4.0, 4.0, 2.5), view((61, 47), (3.5, 3.5), 2.4, off)
    img = np.zeros(61 * 47, np.float32)
    one = img.copy()
    img[20 * 61 + 33], one[20 * 61 + 33] = np.nan, 1.0
    got = np.isnan(P.drr_adjoint(torch.from_numpy(img).cuda(), vol, cb, 1.25).cpu().numpy())
    wt = O.drr_adjoint(one, vol, cb, 1.25)
    # a voxel at the very edge of a sample's support may round either way
    near = np.zeros((19, 31, 35), bool)
    v = (wt > 0).reshape(17, 29, 33)
    for d in np.ndindex(3, 3, 3):
        near[d[0]:d[0] + 17, d[1]:d[1] + 29, d[2]:d[2] + 33] |= v
    assert got[wt > 1e-3].all() and not got[~near[1:-1, 1:-1, 1:-1].ravel()].any()


@pytest.mark.parametrize("off", OFFSETS)
@pytest.mark.parametrize("tile", range(6))
@pytest.mark.parametrize("nz", [9, 18])
def test_gradient_columns(P, nz, tile, off):
    vol, cb = S.volume(70, 37, nz, 4.0, 4.0, 4.0), view((61, 31), (5.0, 5.0), 0.9, off)
    f0, _ = S.phantom(vol, 10.0, seed=5)
    f0 = (f0 * (1 + 0.1 * S.rng(6).uniform(-1, 1, f0.shape))).astype(np.float32)     # no flat tissue
    U = S.eigen_dvfs(vol, 2, seed=7)
    step, w = 2.0, np.array([0.6, -0.3])
    y = O.drr_forward(O.warp_volume(f0, O.pca_dvf(None, U, np.array([0.9, 0.1]), vol), vol), vol, cb, step)
    y = y.astype(np.float32)
    d = P.tuning_get(vol, cb, 2)
    try:
        P.tuning_set(vol, cb, 2, dict(d, voxel_tile=tile))
        J, G, ab = P.cost_grad(torch.from_numpy(f0.ravel()).cuda(), None, torch.from_numpy(U.ravel()).cuda(), w,
                               torch.from_numpy(y).cuda(), vol, cb, step)
    finally:
        P.tuning_clear()
    Jr, Gr, _ = O.cost_grad(f0, None, U, w, y, vol, cb, step)
    assert abs(J - Jr) <= 1e-4 * Jr
    assert np.linalg.norm(G - Gr) <= 1e-3 * np.linalg.norm(Gr)
