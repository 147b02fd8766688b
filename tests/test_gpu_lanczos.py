"""The Lanczos kernels of sp_lowest_mode at the edges of their tiles.

Reference: the same Lanczos recursion, with two Gram-Schmidt passes, in numpy
on the oracle's Hessian-vector product.  Sizes: one spin past a tile of 128
spins, one and several tiles per block (more than 152 tiles), basis sizes below,
at and above the chunks of 16 vectors that one group of a block takes, and past
the 64 vectors of one sweep of all four groups.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _reference(o, n, v, m):
    tangent = lambda w: w - np.sum(w * n, axis=1, keepdims=True) * n  # noqa: E731
    q = tangent(v)
    Q, a, b = [], [], []
    q = q / np.linalg.norm(q)
    for _ in range(m):
        Q.append(q.ravel())
        w = o.hessian_apply(n, q)
        a.append(np.sum(w * q))
        S = np.stack(Q)
        for _ in range(2):
            w = tangent((w.ravel() - S.T @ (S @ w.ravel())).reshape(n.shape))
        b.append(np.linalg.norm(w))
        q = w / b[-1]
    lam, V = np.linalg.eigh(np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1))
    y = V[:, 0] @ np.stack(Q)
    return lam[0], y / np.linalg.norm(y), np.abs(lam).max(), lam[1] - lam[0]


# the last lattice has 153 tiles: block 0 takes two of them
@pytest.mark.parametrize("dims,m", [((129, 1), 15), ((43, 3), 16), ((60, 37), 17), ((40, 40), 80), ((139, 140), 33)])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_lowest_ritz_pair_matches_reference(dims, m, prec):
    g = I.hexagonal(*dims, periodic=(True, dims[1] > 2), mu_s=2.0)
    h = dict(J=[1.0, 0.1], dmi_kind="interfacial", D=[0.3], K=[0.1], Khat=[[0.2, 0, 1]], B=[0.1, 0, 0.7])
    o = oracle.System(g, h)
    c = B.Context(g, h, prec)
    n0, v0 = I.random_spins(c.N, 3), np.random.default_rng(4).standard_normal((c.N, 3))
    if prec == "f32":
        n0, v0 = n0.astype(np.float32).astype(np.float64), v0.astype(np.float32).astype(np.float64)
    lam, mode = c.lowest_mode(c.spins(n0), c.spins(v0), m)
    ref, y, scale, gap = _reference(o, n0, v0, m)
    # records of precision u: the operator, m vectors and their products are
    # each off by a few u |H|, the vector by that over the gap
    u = 1.2e-16 if prec == "f64" else 6e-8
    assert abs(lam - ref) <= 64 * m * u * scale
    x = mode[:, :3].double().cpu().numpy().ravel()
    assert min(np.linalg.norm(x - y), np.linalg.norm(x + y)) <= 64 * m * u * scale / gap + 8 * u
    assert torch.all(mode[:, 3] == 0)
