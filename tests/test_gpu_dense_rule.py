"""The choice between the two gradient kernels (the gather at the compacted
voxels and the walk over voxel columns).  On a checkerboard of blocks every
group of columns holds compacted voxels, whatever their share, so the columns
cost the same at 6 % as at 15 %, while the gather's cost is proportional to the
voxels.  From blocks of 48 voxels (always the gather) to blocks of 20 the
gradient pass may therefore grow by no more than the number of compacted voxels
does; 1.25 times that is allowed for the clock and the caches (the columns
there: 1.7 times).  And the choice changes no gradient beyond rounding: cached
and computed weights give the same bits on a CT with texture, and the two
kernels' gradients agree with the FP64 oracle as in the other tests (1e-4)."""
import numpy as np
import pytest

import cases
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


def checkerboard(n, p):
    x, y, z = (torch.arange(m, device="cuda") // p for m in n)
    odd = (z[:, None, None] + y[None, :, None] + x[None, None, :]) % 2
    return (0.01 + 0.01 * odd).reshape(-1).float()


def compacted(n, p):
    """Cells [i, i + 1) with a block's face inside, on the grid's inside."""
    inner = [sum(1 for i in range(m - 1) if (i + 1) % p) for m in n]
    return np.prod(n) - np.prod(inner)


def test_gather_where_columns_do_not_pay(P):
    n = (256, 256, 100)
    vol = S.volume(*n, 1.75, 1.7, 2.5)
    cb = S.cone_beam(512, 384, 0.78, 0.78, 0.8, off_u=6.0, off_v=-7.0)
    vs, cs = P.vol_struct(vol), P.cb_struct(cb)
    ws = P.Workspace(vs, cs, 1)
    U = torch.ones(3 * n[0] * n[1] * n[2], device="cuda")          # the same shift everywhere, 0.3 mm
    y = torch.rand(512 * 384, device="cuda", generator=torch.Generator("cuda").manual_seed(2))

    def ms(f0):
        times = []
        for _ in range(6):
            P.profile(True)
            P.cost_grad(f0, None, U, [0.3], y, vs, cs, 0.8, ws=ws)
            torch.cuda.synchronize()
            times.append(P.profile_read()["adjoint_grad"][1])
            P.profile(False)
        return min(times[1:])

    few, many = compacted(n, 48), compacted(n, 20)
    assert few * 8 < np.prod(n) <= many * 8
    assert ms(checkerboard(n, 20)) <= 1.25 * many / few * ms(checkerboard(n, 48))


@pytest.mark.parametrize("kind", ["texture", "checkerboard"])
@pytest.mark.parametrize("off_v", [0.0, -9.0])
def test_gradients_and_fixed_view(P, kind, off_v):
    n = (72, 66, 40)
    pb = cases.make_problem((*n, 4.0, 4.0, 4.0), 2, (129, 97, 3.1, 3.1), 0.7, (0.8, -0.3), off=(3.0, off_v))
    if kind == "texture":
        pb["f0"] = (pb["f0"] * S.rng(9).uniform(0.9, 1.1, pb["f0"].shape)).astype(np.float32)
    else:
        pb["f0"] = checkerboard(n, 9).cpu().numpy().reshape(pb["f0"].shape)
    d = cases.to_dev(pb)
    w = np.array([0.5, -0.2])
    J, G, _ = P.cost_grad(d["f0"], None, d["U"], w, d["y"], pb["vol"], pb["cb"], pb["step"])
    Jo, Go, _ = O.cost_grad(pb["f0"], None, pb["U"], w, pb["y"], pb["vol"], pb["cb"], pb["step"])
    assert abs(J - Jo) <= 1e-4 * Jo and np.abs(G - Go).max() <= 1e-4 * np.abs(Go).max()
    sv = P.Solver(d["f0"], None, d["U"], pb["vol"], pb["cb"], P.default_params(pb["step"], max_iter=3))
    plain = sv.solve(d["y"], np.zeros(2))
    sv.fix_view(0.7)
    cached = sv.solve(d["y"], np.zeros(2))
    host = P.solve_projection(d["f0"], None, d["U"], d["y"], pb["vol"], pb["cb"], np.zeros(2),
                              P.default_params(pb["step"], max_iter=3))
    for got in (cached, host):
        assert np.array_equal(plain[0], got[0]) and plain[1] == got[1]
    sv.close()
