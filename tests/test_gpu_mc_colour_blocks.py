"""Colours of few spins: blocks of one replica's trials, and blocks of several replicas'.

Which of the two a sweep takes depends on the number of replicas; a replica's spins,
cone and accepted trials do not.
"""
import numpy as np
import pytest
import torch

from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# 400 replicas pack (17^3: 17 colours of 289 spins, 15^3: 3 of 1125, 6^3: 2 of 108, 8 x 6 x
# 4 with two shells: more colours of less), 3 do not
@pytest.mark.parametrize("dims,J", [((17, 17, 17), [1.0]), ((15, 15, 15), [1.0]), ((6, 6, 6), [1.0]), ((8, 6, 4), [1.0, 0.2])])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("sample", [False, True])
def test_replicas_do_not_depend_on_the_batch(dims, J, prec, sample):
    R, few, sweeps = 400, 3, 18
    out = []
    for n_rep in (R, few):
        c = B.Context(I.simple_cubic(*dims), dict(J=J), prec)
        c.set_option("mc_resident", 0)
        x = c.spins(np.stack([I.random_spins(c.N, r % few) for r in range(n_rep)]))
        T = [5.0 + 4.0 * (r % few) for r in range(n_rep)]
        cone, st = c.mc_sweeps(x, T, sweeps, seed=3, sweep0=9, sample=sample)[:2]
        assert c.sync_status()[0] == 0
        out.append((x, cone, st[:, 5:], st[:, :5]))
    for a, b in zip(out[0][:3], out[1][:3]):
        assert torch.equal(a[:few], b)
    # the same sums in another order: twenty float-float additions, 2^-47 each, of
    # magnetisations that cancel to a hundredth
    assert torch.allclose(out[0][3][:few], out[1][3], rtol=1e-10, atol=0)
