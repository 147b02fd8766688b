"""A GNEB call with the layout of the call before launches kernels only: it can be
captured, from whatever depth of the caller's stack it is made."""
import numpy as np
import pytest
import torch

from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import inputs as I

pytestmark = pytest.mark.gpu

H = dict(J=[1.0], dmi_kind="interfacial", D=[0.3], K=[0.1], Khat=[[0, 0, 1]], B=[0, 0, 0.7])


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_repeated_call_can_be_captured(prec):
    c = B.Context(I.hexagonal(20, 17, periodic=(True, True)), H, prec)
    M = 5
    x0 = c.spins(np.stack([I.perturbed(I.ferromagnet(c.N, (0.3 * m, 0, 1.0)), 0.2, m) for m in range(M)]))

    def step(x, v):
        return c.gneb_step(x, v, n_iter=3, dt=0.05)

    x, v = x0.clone(), torch.zeros_like(x0)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        step(x, v)
        step(x, v)  # the same chain twice: what a replay has to give
        want = (x.clone(), v.clone())
        y, w = x0.clone(), torch.zeros_like(x0)
        step(y, w)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            (lambda: (lambda: step(y, w))())()
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, want[0]) and torch.equal(w, want[1])
    assert c.sync_status()[0] == 0
