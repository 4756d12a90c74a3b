"""dJ/df0 at extreme magnitudes: the scatter's power-of-two scale covers images
whose residuals are tiny or huge.  Scaling the image and the CT together by a
power of two s scales J by s^2 and dJ/df0 by s, exactly in float arithmetic, so
the gradients must agree to the scatter's fixed-point step (2^-40 of the
largest contribution, far below the float rounding of the result)."""
import numpy as np
import pytest

from paper_1102_1712_gb300 import synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dims", [(33, 30, 9), (36, 29, 10)])
@pytest.mark.parametrize("power", [-60, -7, 40])
def test_grad_f0_scale(dims, power):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1102_1712_gb300 import build as B
    from paper_1102_1712_gb300 import pcasolve as P
    B.build()
    vol, cb = S.volume(*dims, 4.0, 4.0, 4.0), S.cone_beam(41, 25, 5.0, 5.0, 0.3)
    g = S.rng(3)
    f0 = torch.from_numpy(g.uniform(0.0, 0.03, np.prod(dims)).astype(np.float32)).cuda()
    U = torch.from_numpy(S.eigen_dvfs(vol, 2, seed=4).ravel()).cuda()
    y = P.drr_forward(f0, vol, cb, 2.0) + 0.01 * torch.from_numpy(g.standard_normal(1025).astype(np.float32)).cuda()
    w, s = np.array([0.4, -0.2]), 2.0 ** power
    ref = P.cost_grad_f0(f0, None, U, w, y, vol, cb, 2.0)[3].double()
    got = P.cost_grad_f0(f0 * s, None, U, w, y * s, vol, cb, 2.0)[3].double() / s
    # J is also computed on its own (rows that the fused warp takes, and the others)
    J = P.cost_grad_f0(f0, None, U, w, y, vol, cb, 2.0, want_grad=False, want_grad_f0=False)[0]
    assert J == P.cost_grad_f0(f0, None, U, w, y, vol, cb, 2.0)[0]
    assert float((got - ref).abs().max()) <= 1e-6 * float(ref.abs().max())
