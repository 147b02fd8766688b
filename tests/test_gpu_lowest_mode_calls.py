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


@pytest.mark.parametrize("prec,exponents", [("f32", (-100, -80, 70, 120)), ("f64", (-900, -600, 550, 1000))])
def test_start_vectors_of_any_size(prec, exponents):
    # a power of two changes no rounding of the run: the same bits
    c, (n, _), v = _system(40, prec)
    lam, mode = c.lowest_mode(n, v.clone(), 24)
    seeded = c.lowest_mode(n, torch.zeros_like(v), 24)[1]
    assert not torch.equal(mode, seeded)
    for e in exponents:
        l2, m2 = c.lowest_mode(n, v * 2.0 ** e, 24)
        assert l2 == lam and torch.equal(m2, mode), e


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_start_vector_that_is_not_finite(prec):
    # infinite: reported; NaN: replaced, as a zero one is
    c, (n, _), v = _system(40, prec)
    w = v.clone()
    w[7, 1] = float("inf")
    with pytest.raises(B.SpinError):
        c.lowest_mode(n, w, 8)
    w[7, 1] = float("nan")
    assert torch.equal(c.lowest_mode(n, w, 8)[1], c.lowest_mode(n, torch.zeros_like(v), 8)[1])
