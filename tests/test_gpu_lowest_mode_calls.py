"""sp_lowest_mode as a call: what it leaves on the stream, and the start vectors it takes."""
import numpy as np
import pytest
import torch

from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import inputs as I

pytestmark = pytest.mark.gpu

H = dict(J=[1.0], dmi_kind="interfacial", D=[0.3], K=[0.1], Khat=[[0, 0, 1]], B=[0, 0, 0.7])


def _system(n, prec):
    c = B.Context(I.hexagonal(n, n, periodic=(True, True), mu_s=2.0), H, prec)
    return c, [c.spins(I.random_spins(c.N, k)) for k in (1, 2)], c.spins(np.random.default_rng(3).standard_normal((c.N, 3)))


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_returns_with_nothing_left_on_the_stream(prec):
    # the last launches read the context's scratch (64 vectors of 512 x 512 spins:
    # a tenth of a millisecond): a call on another stream may follow at once
    c, (n, _), v = _system(512, prec)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        for _ in range(3):
            m = v.clone()
            c.lowest_mode(n, m, 64)
            assert s.query()


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_two_streams_give_the_modes_of_single_calls(prec):
    c, states, v = _system(96, prec)
    single = [c.lowest_mode(n, v.clone(), 24) for n in states]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(5):
        out = []
        for s, n in zip(streams, states):
            m = v.clone()
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(s):
                out.append(c.lowest_mode(n, m, 24))
        torch.cuda.synchronize()
        for (lam, m), (l0, m0) in zip(out, single):
            assert lam == l0 and torch.equal(m, m0)
