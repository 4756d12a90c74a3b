"""warp_volume on rows of any length: values against the FP64 oracle on both
sides of the size from which a thread takes two voxels (an odd voxel count
among them, so that the last thread has one), 5e-5 of the maximum as in the
other warp tests, whose extents are below 256, and more in proportion to larger
ones (a position's rounding); and the time per voxel, which must not depend on whether the
rows are a multiple of a warp: 400x360x100 against 384x360x100 has the same
work per voxel, so the ratio is 1 but for the lanes and tests that a launch
wastes on its rows' ends (1.25 with blocks that end with the row); the line is
about half of that."""
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


@pytest.mark.parametrize("dims", [(131, 13, 9), (257, 130, 129), (401, 151, 101), (5, 1151, 1150)])
def test_values(P, dims):
    vol = S.volume(*dims, 2.0, 3.0, 2.5)
    g = S.rng(4)
    f0 = g.uniform(0.0, 0.03, np.prod(dims)).astype(np.float32)
    dvf = g.uniform(-6.0, 6.0, 3 * f0.size).astype(np.float32)
    got = P.warp_volume(torch.from_numpy(f0).cuda(), torch.from_numpy(dvf).cuda(), vol).cpu().numpy()
    ref = O.warp_volume(f0.reshape(dims[::-1]), dvf.reshape(3, -1), vol)
    assert np.abs(got - ref.ravel()).max() <= 5e-5 * max(1.0, max(dims) / 256) * f0.max()


def test_time_per_voxel_of_ragged_rows(P):
    def problem(nx):
        vol = P.vol_struct(S.volume(nx, 360, 100, 2.0, 2.0, 2.5))
        n = nx * 360 * 100
        x, y, z = (torch.arange(m, device="cuda", dtype=torch.float32) for m in (nx, 360, 100))
        bump = (torch.sin(z / 16)[:, None, None] + torch.sin(y / 19)[None, :, None] + torch.sin(x / 23)[None, None, :]).reshape(-1)
        dvf = torch.cat([4.0 * bump, -3.0 * bump, 5.0 * bump])
        f0 = torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        return vol, f0, dvf, torch.empty_like(f0), n

    def ns_per_voxel(q):
        vol, f0, dvf, out, n = q
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(10):
            P.warp_volume(f0, dvf, vol, out=out)
        b.record()
        b.synchronize()
        return a.elapsed_time(b) * 1e5 / n

    even, ragged = problem(384), problem(400)
    times = [(ns_per_voxel(even), ns_per_voxel(ragged)) for _ in range(12)][2:]
    assert min(t[1] for t in times) <= 1.14 * min(t[0] for t in times)
