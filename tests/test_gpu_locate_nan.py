"""localize_tumor where the field is not a number: an update that is NaN counts as
no change, in one component or in all, on the first iterate or a later one, as
the FP64 oracle's fmax has it.  Centroids 1e-6 mm, as in the other tests."""
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


@pytest.mark.parametrize("bad,where", [((0,), "everywhere"), ((0, 1), "everywhere"), ((0, 1, 2), "everywhere"),
                                       ((0,), "second iterate"), ((2,), "second iterate"),
                                       ((0, 1, 2), "second iterate")])
def test_nan_field(P, bad, where):
    vol = S.volume(11, 9, 7, 4.0, 4.0, 4.0)
    U = np.zeros((1, 3, 7, 9, 11), np.float32)
    U[:, 0] = 6.0                                   # one step of -6 mm along x, 1.5 voxels
    for c in bad:
        if where == "everywhere":
            U[:, c] = np.nan
        else:
            U[:, c, :, :, :5] = np.nan              # voxels left of the start's cell
    at = np.array([0.7, 0.9, -1.1])
    c, ok = P.localize_tumor(None, torch.from_numpy(U.ravel()).cuda(), np.ones(1), vol, at)
    co, oko = O.localize_tumor(None, U.reshape(1, 3, -1), np.ones(1), vol, at)
    assert ok == oko
    assert np.array_equal(np.isnan(c), np.isnan(co)) and np.nanmax(np.abs(np.nan_to_num(c) - np.nan_to_num(co))) <= 1e-6
