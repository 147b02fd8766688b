"""Which kernels a batch of replicas takes by itself, and what that means for its bits.

A batch stays on the 27-point path where the general passes' split gives a CTA eight
planes or more (all replicas' planes over one wave of CTAs) or the lean passes are
faster, and then gives every replica the bits of a call on it alone; smaller
batches take the per-spin kernels, which agree with that call within FP32 rounding
(the bound of test_gpu_lean.py for five steps).
"""
import numpy as np
import pytest
import torch

from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SC = I.cfg_sc_128(4)["hamiltonian"]


def _run(dims, R, solver, steps, h=SC, **options):
    c = B.Context(I.simple_cubic(*dims), h, "f32")
    for k, v in options.items():
        c.set_option(k, v)
    temps = [2.0 * r for r in range(R)]
    n0 = c.spins(np.stack([I.random_spins(c.N, 40 + r) for r in range(R)]))
    kw = dict(solver=solver, dt=1e-3, alpha=0.1, seed=5, step0=7)
    x = n0.clone()
    c.llg_step_replicas(x, temps, steps, replica=3, **kw)
    y = n0.clone()
    for r in {0, 1, R // 2, R - 1}:
        c.llg_step(y[r], steps, T=temps[r], replica=3 + r, **kw)
        yield x[r], y[r]


@pytest.mark.parametrize("dims,R", [((16, 16, 16), 256), ((22, 22, 22), 60), ((30, 30, 30), 12), ((32, 32, 32), 29)])
def test_large_batches_give_the_bits_of_single_calls(dims, R):
    for x, y in _run(dims, R, "heun", 5):
        assert torch.equal(x, y)


@pytest.mark.parametrize("dims,R", [((22, 22, 22), 8), ((30, 30, 30), 4), ((16, 16, 16), 29)])
def test_small_batches_agree_within_rounding(dims, R):
    for x, y in _run(dims, R, "heun", 5):
        assert (x - y).abs().max().item() <= 2e-6


# the general passes of a batch, reached by option
@pytest.mark.parametrize("solver", ["heun", "depondt"])
@pytest.mark.parametrize("lean", [0, 1])
def test_batches_of_either_family_give_the_bits_of_single_calls(solver, lean):
    for x, y in _run((13, 11, 9), 5, solver, 4, small_path=0, planes_per_cta=3, cubic_lean=lean):
        assert torch.equal(x, y)
