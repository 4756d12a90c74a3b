"""The incoming gradient of pca_cost belongs to the caller again when backward
returns, also where it lies in pinned memory and the stream still has work: the
product for f0 must have its value by then."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_incoming_gradient_is_read_before_backward_returns(monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1102_1712_gb300 import autograd as A
    from paper_1102_1712_gb300 import build as B
    from paper_1102_1712_gb300 import pcasolve as P
    B.build()
    pb = cases.make_problem((24, 22, 12, 6.0, 6.0, 6.0), 2, (31, 23, 8.0, 8.0), 0.4, (0.8, -0.3))
    d = cases.to_dev(pb)
    prob = A.problem(d["U"], d["y"], P.vol_struct(pb["vol"]), P.cb_struct(pb["cb"]), pb["step"])

    def gradient(busy):
        f0 = d["f0"].clone().requires_grad_(True)
        J = A.pca_cost(torch.tensor([0.5, -0.2]), f0, prob)
        gJ = torch.full((), 3.0, dtype=torch.float64, pin_memory=True)
        if busy:
            call = P.cost_grad_f0

            def call_then_work(*a, **kw):
                r = call(*a, **kw)
                torch.cuda._sleep(200_000_000)          # about 0.1 s on the stream before the product
                return r

            monkeypatch.setattr(P, "cost_grad_f0", call_then_work)
        J.backward(gJ)
        gJ.fill_(0.0)
        torch.cuda.synchronize()
        return f0.grad

    want = gradient(False)
    assert float(want.abs().max()) > 0
    assert torch.equal(gradient(True), want)
