"""drr_siddon where float cannot hold a ray's sum in voxel units, or the step from
one voxel to the next, but can hold the path in mm: the same result as with
values smaller by a power of two, scaled back.  Tolerance 1e-6 of the maximum,
as in the other Siddon tests."""
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


@pytest.mark.parametrize("signs", [False, True])
@pytest.mark.parametrize("angle", [0.0, 0.8])
def test_large_values(P, signs, angle):
    n = (60, 52, 12)
    vol, cb = S.volume(*n, 0.02, 0.02, 0.02), S.cone_beam(31, 9, 0.06, 0.05, angle, off_u=0.017, off_v=0.013)
    g = S.rng(3)
    f = g.uniform(1.0, 2.0, n[::-1])
    if signs:                                   # neighbours of opposite sign: their difference overflows
        f *= g.choice([-1.0, 1.0], f.shape)
    f = f.astype(np.float32)
    p = P.drr_siddon(torch.from_numpy((f * np.float32(2.0 ** 126)).ravel()).cuda(), vol, cb).cpu().numpy()
    po = O.siddon_forward(f.astype(np.float64), vol, cb)
    assert np.abs(po).max() > 0.1 and np.abs(p.astype(np.float64) * 2.0 ** -126 - po).max() <= 1e-6 * np.abs(po).max()
