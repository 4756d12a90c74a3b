"""The autotuner leaves the batch projector's chunk alone on a detector whose batch
stages nothing (all chunks are the same work there, and the entry also serves
larger detectors of its bucket), and still chooses its patch width."""
import numpy as np
import pytest

from cases import make_problem, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_chunk_of_a_split_batch_stays():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1102_1712_gb300 import build as B
    from paper_1102_1712_gb300 import pcasolve as P
    B.build()
    pb = make_problem((40, 36, 20, 6.0, 6.0, 6.0), 2, (90, 70, 4.0, 4.0), 0.4, np.array([0.7, -0.4]))
    d = to_dev(pb)
    P.tuning_clear()
    try:
        t = dict(P.tuning_get(pb["vol"], pb["cb"], 2), chunk=[40, 6, 10, 64, 2, 30, 50, 8])
        P.tuning_set(pb["vol"], pb["cb"], 2, t)
        got = P.autotune(d["f0"], None, d["U"], d["y"], pb["vol"], pb["cb"], P.default_params(pb["step"]))
        assert got["chunk"] == t["chunk"] and all(2 <= v <= 4 for v in got["ray_lw4"])
    finally:
        P.tuning_clear()
