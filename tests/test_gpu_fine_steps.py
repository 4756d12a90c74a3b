"""P^T where the sample indices leave the range in which an addition rounds them to
whole numbers exactly (2^22): tens of thousands of samples a voxel.  A voxel's
sum has n = 2 voxels / step terms, each rounded to 2^-24, so n 2^-24 of the
maximum is allowed."""
import numpy as np
import pytest

import oracle as O
from paper_1102_1712_gb300 import synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("step", [4e-4, 1.7e-4, 1.1e-4, 5e-5])
@pytest.mark.parametrize("off_v", [0.0, 0.7])
def test_adjoint_of_fine_steps(step, off_v):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1102_1712_gb300 import build as B
    from paper_1102_1712_gb300 import pcasolve as P
    B.build()
    vol, cb = S.volume(5, 4, 3, 2.0, 2.0, 2.0), S.cone_beam(6, 5, 2.5, 2.0, 0.6, off_v=off_v)
    img = S.rng(8).uniform(0.5, 1.5, 30).astype(np.float32)
    got = P.drr_adjoint(torch.from_numpy(img).cuda(), vol, cb, step).cpu().numpy()
    ref = O.drr_adjoint(img.reshape(5, 6).astype(np.float64), vol, cb, step).ravel()
    err = np.abs(got - ref).max() / np.abs(ref).max()
    print(f"step {step}: error {err:.2e} of the maximum, allowed {4.0 / step * 2.0 ** -24:.2e}")
    assert err <= 4.0 / step * 2.0 ** -24
