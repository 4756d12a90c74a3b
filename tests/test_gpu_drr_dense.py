"""drr_forward against the FP64 oracle at the edges of its ray patches, window
parts and inner box: detectors that no patch divides, windows shorter than the
parts, volumes without an inner box, rays half outside, each patch width.
Tolerance: 1e-4 of the maximum, as in the other projector tests."""
import numpy as np
import pytest

import oracle as O
from paper_1102_1712_gb300 import synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [((32, 33, 17, 4.0, 4.0, 4.0), (33, 21, 5.0, 5.0), 0.2, (0.0, 0.0), 2.0),       # 16 wide
         ((32, 33, 17, 4.0, 4.0, 4.0), (33, 21, 5.0, 5.0), 1.26, (0.0, 0.0), 2.0),      # 8
         ((32, 33, 17, 4.0, 4.0, 4.0), (33, 21, 5.0, 5.0), np.pi / 2, (0.0, 0.0), 2.0),  # 4
         ((61, 40, 23, 4.0, 4.0, 4.0), (17, 5, 5.0, 5.0), 4.0, (90.0, -30.0), 2.0),     # rays half outside
         ((2, 2, 2, 30.0, 30.0, 30.0), (19, 13, 5.0, 5.0), 0.7, (0.0, 0.0), 15.0),      # a few samples a ray
         ((1, 9, 3, 40.0, 4.0, 4.0), (19, 13, 5.0, 2.0), 0.7, (0.0, 0.0), 2.0),         # no inner box
         ((40, 38, 20, 3.0, 3.0, 3.0), (1, 37, 5.0, 3.0), 0.0, (0.0, 0.0), 0.3),        # long windows
         ((40, 38, 20, 3.0, 3.0, 3.0), (37, 1, 3.0, 5.0), 2.9, (0.0, 0.0), 9.0)]


@pytest.mark.parametrize("dims,det,angle,off,step", CASES)
def test_drr_dense(dims, det, angle, off, step):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1102_1712_gb300 import build as B
    from paper_1102_1712_gb300 import pcasolve as P
    B.build()
    vol = S.volume(*dims)
    f = S.rng(3).uniform(0.0, 0.03, dims[0] * dims[1] * dims[2]).astype(np.float32)
    cb = S.cone_beam(det[0], det[1], det[2], det[3], angle, off_u=off[0], off_v=off[1])
    got = P.drr_forward(torch.from_numpy(f).cuda(), vol, cb, step).cpu().numpy().astype(np.float64)
    ref = O.drr_forward(f, vol, cb, step)
    assert np.abs(got - ref).max() <= 1e-4 * max(np.abs(ref).max(), 1e-30)
