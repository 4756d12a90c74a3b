"""drr_forward where rays are short and many: values on both sides of the lines
between a thread per ray, four and eight warps a patch against the FP64 oracle
(1e-4 of the maximum, as in the other DRR tests), and two times on the same large
detector, of what have alike a ray's set-up, once a warp.  48 voxels across
against 128, 2.7 times the samples: 0.44 with four warps a patch, 0.49 with eight,
which is more than one thread a ray takes; the line is between.  8 voxels across
against 48: 0.47 with a thread per ray, 0.71 with eight warps a patch."""
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


@pytest.mark.parametrize("det", [(37, 21), (199, 131), (259, 255)])
@pytest.mark.parametrize("dims", [(1, 1, 1), (9, 13, 5), (32, 21, 7), (45, 44, 3)])
def test_values(P, dims, det):
    vol = S.volume(*dims, 160.0 / dims[0], 150.0 / dims[1], 60.0 / dims[2])
    cb = S.cone_beam(det[0], det[1], 300.0 / det[0], 150.0 / det[1], 0.9, off_u=11.0, off_v=-6.0)
    step = 0.5 * min(vol["sx"], vol["sy"], vol["sz"])
    f = S.rng(5).uniform(0.0, 0.03, np.prod(dims)).astype(np.float32)
    p = P.drr_forward(torch.from_numpy(f).cuda(), vol, cb, step).cpu().numpy()
    po = O.drr_forward(f.reshape(dims[::-1]), vol, cb, step).ravel()
    assert po.max() > 0 and np.abs(p.ravel() - po).max() <= 1e-4 * po.max()


def test_time_of_short_rays(P):
    def problem(n):
        s = (450.0 / n[0], 420.0 / n[1], 240.0 / n[2])
        f = torch.rand(n[0] * n[1] * n[2], device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        return f, P.vol_struct(S.volume(*n, *s)), P.cb_struct(S.cone_beam(1024, 768, 0.38, 0.38, 0.3)), 0.5 * min(s)

    def ms(q):
        f, vol, cb, step = q
        out = torch.empty(1024 * 768, device="cuda")
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(10):
            P.drr_forward(f, vol, cb, step, out=out)
        b.record()
        b.synchronize()
        return a.elapsed_time(b)

    q = [problem(n) for n in ((8, 8, 8), (48, 44, 24), (128, 128, 64))]
    t = np.min([[ms(p) for p in q] for _ in range(10)][2:], axis=0)
    assert t[1] <= 0.475 * t[2] and t[0] <= 0.59 * t[1], t
