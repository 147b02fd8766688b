"""The sums over an image's blocks at the edges of the rows its last block adds.

One iteration of the minimiser from rest gives v = c F with c = v.F / F.F over all
spins, and the largest |F|; an iteration of GNEB the energies of its images.  The
reference takes both from 64-bit fields of the states before and after.  The field
of the FP32 kernels is within 16 roundings of the sum of its terms (below 8 meV
here), 8e-6 against forces of order 1: c and max |F| are good to 2e-5.  A block left
out of 4100 changes c by 2e-4.
"""
import numpy as np
import pytest
import torch

from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import inputs as I

pytestmark = pytest.mark.gpu

H = dict(J=[1.0], dmi_kind="interfacial", D=[0.3], K=[0.1], Khat=[[0, 0, 1]], B=[0, 0, 0.7])
# blocks of 256 spins: 1, 31, 32, 34, 129, 1026, 4100
DIMS = [(9, 11), (256, 31), (256, 32), (257, 33), (256, 129), (512, 513), (1024, 1025)]


def _force(ref, x):
    x = x.double()
    b = ref.effective_field(x)
    b[:, 3] = 0
    x = torch.cat([x[:, :3], torch.zeros_like(x[:, :1])], 1)
    return b - (b * x).sum(1, keepdim=True) * x


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec,tol", [("f32", 2e-5), ("f64", 1e-12)])
@pytest.mark.parametrize("batch", [False, True])
def test_projection_and_largest_force(dims, prec, tol, batch):
    g = I.square(*dims, periodic=(True, True))
    c, ref = B.Context(g, H, prec), B.Context(g, H, "f64")
    x = c.spins(I.random_spins(c.N, 2))
    v, dt = torch.zeros_like(x), 0.1
    f0 = _force(ref, x)
    if batch:
        it, mt = B.minimise_batch([c], x, v, [0], dt=dt, tol=1e-12, max_iter=1)
        it, mt = it[0], mt[0]
    else:
        it, mt = c.minimise(x, v, dt=dt, tol=1e-12, max_iter=1)
    assert it == 1
    f1 = _force(ref, x)
    w = 0.5 * dt * (f0 + f1)
    coef = (w * f1).sum() / (f1 * f1).sum()
    assert coef > 0
    assert (v.double() - coef * f1).abs().max() <= tol * (coef * f1).norm(dim=1).max()
    top = f1.norm(dim=1).max().item()
    assert abs(mt - top) <= tol * top


@pytest.mark.parametrize("dims,M", [((9, 11), 3), ((257, 33), 5), ((512, 513), 4), ((1024, 1025), 3)])
@pytest.mark.parametrize("prec,tol", [("f32", 1e-5), ("f64", 1e-12)])
def test_image_energies(dims, M, prec, tol):
    g = I.square(*dims, periodic=(True, True))
    c, ref = B.Context(g, H, prec), B.Context(g, H, "f64")
    x = torch.stack([c.spins(I.perturbed(I.ferromagnet(c.N, (0.1 * m, 0, 1.0)), 0.2, m)) for m in range(M)])
    E, F = c.gneb_step(x, torch.zeros_like(x), n_iter=1, dt=0.02)
    want = torch.stack([ref.energy(x[m].double())[0] for m in range(M)])
    assert ((E.double() - want).abs() <= tol * want.abs()).all()
