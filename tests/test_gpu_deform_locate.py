"""warp_volume and localize_tumor against the FP64 oracle where their rewritten
loops can go wrong: rows of one voxel, shorter and longer than a block, fields
that leave the grid or are not finite; iterates that change cells, sit on a
voxel, start outside the grid, or have taps without weight that are not finite.
Tolerances: warp 5e-5 of the maximum (as in the other warp tests), centroid
1e-6 mm (the fixed point's own)."""
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


@pytest.mark.parametrize("dims", [(1, 7, 5), (2, 2, 2), (31, 5, 4), (65, 3, 3), (513, 3, 2), (1025, 2, 2)])
def test_warp_rows(P, dims):
    vol = S.volume(*dims, 2.0, 3.0, 2.5)
    g = S.rng(1)
    f0 = g.uniform(0.0, 0.03, np.prod(dims)).astype(np.float32)
    dvf = g.uniform(-6.0, 6.0, 3 * f0.size).astype(np.float32)
    got = P.warp_volume(torch.from_numpy(f0).cuda(), torch.from_numpy(dvf).cuda(), vol).cpu().numpy()
    ref = O.warp_volume(f0.reshape(dims[::-1]), dvf.reshape(3, -1), vol)
    assert np.abs(got - ref.ravel()).max() <= 5e-5 * f0.max()
    dvf[::3] = np.nan                       # a position that is not a number lies outside
    got = P.warp_volume(torch.from_numpy(f0).cuda(), torch.from_numpy(dvf).cuda(), vol).cpu().numpy()
    bad = np.isnan(dvf.reshape(3, -1)).any(axis=0)
    assert (got[bad] == 0.0).all() and np.isfinite(got).all()


def test_localize_cells(P):
    vol = S.volume(19, 17, 13, 4.0, 4.0, 4.0)
    N = 19 * 17 * 13
    U = (0.35 * S.eigen_dvfs(vol, 2, seed=5, sigma_mm=9.0)).astype(np.float32)
    dU = torch.from_numpy(U.ravel()).cuda()
    g = S.rng(2)
    for _ in range(12):
        w, c_ref = g.uniform(-2.0, 2.0, 2), g.uniform(-40.0, 40.0, 3)
        c, ok = P.localize_tumor(None, dU, w, vol, c_ref)
        co, oko = O.localize_tumor(None, U, w, vol, c_ref)
        assert ok == oko and (not ok or np.abs(c - co).max() <= 1e-6)
    # on a voxel, the other taps of its cell not finite and without weight
    bad = np.full((1, 3, N), np.nan, np.float32)
    v = (6 * 17 + 8) * 19 + 9
    bad[:, :, v] = 0.0
    at = np.array([vol["ox"] + 9 * 4.0, vol["oy"] + 8 * 4.0, vol["oz"] + 6 * 4.0])
    c, ok = P.localize_tumor(None, torch.from_numpy(bad.ravel()).cuda(), np.ones(1), vol, at)
    assert ok and np.array_equal(c, at)
    # outside the grid the field is zero
    far = np.array([500.0, -500.0, 500.0])
    c, ok = P.localize_tumor(None, dU, np.ones(2), vol, far)
    assert ok and np.array_equal(c, far)
