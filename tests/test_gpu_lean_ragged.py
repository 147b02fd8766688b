"""The lean FP32 Heun passes on lattices that are not cut into whole column tiles,
and on batches of replicas.

* one step against the oracle, five against the general 27-point passes (the
  bounds of test_gpu_lean.py, whose lattices are whole tiles);
* the same bits for one and two columns per thread and for every split of the
  (tile, plane) units, among them the one taken by itself (runs that do not
  cross tiles);
* replicas in one batch, replayed from a graph or not, give each what a call on
  it alone gives.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import build
from paper_1901_11350_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    B.lib()


SC = I.cfg_sc_128(4)["hamiltonian"]
OPEN = dict(J=[1.0, -0.2], dmi_kind="bulk", D=[0.3], K=[0.1], Khat=[[0.3, 0.1, 1.0]], B=[0.1, -0.2, 1.0])
CASES = {
    "33x16x4_periodic": (I.simple_cubic(33, 16, 4), SC),
    "31x7x5_interfacial_open_y": (I.simple_cubic(31, 7, 5, periodic=(True, False, True)),
                                  dict(J=[1.0], dmi_kind="interfacial", D=[0.25], K=[0.05], Khat=[[0, 0, 1]])),
    "64x9x3_no_dmi": (I.simple_cubic(64, 9, 3), dict(J=[1.0, 0.1, -0.05], K=[0.05], Khat=[[0, 0, 1]])),
    "65x17x6_open": (I.simple_cubic(65, 17, 6, periodic=(False, False, False)), OPEN),
    "2x3x2_periodic": (I.simple_cubic(2, 3, 2), SC),
    "1x9x7_open_x": (I.simple_cubic(1, 9, 7, periodic=(False, True, True)), SC),
    "40x24x1_film": (I.square(40, 24, periodic=(True, False)), dict(J=[1.0], dmi_kind="interfacial", D=[0.3],
                                                                     K=[0.1], Khat=[[0, 0, 1]], B=[0, 0, 1.0])),
}


def _ctx(g, h, lean=1, **options):
    c = B.Context(g, h, "f32")
    c.set_option("small_path", 0)
    c.set_option("cubic_lean", lean)
    for k, v in options.items():
        c.set_option(k, v)
    return c


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("T", [0.0, 10.0])
def test_ragged_step_matches_oracle_and_general_passes(name, T):
    g, h = CASES[name]
    o = oracle.System(g, h)
    n0 = I.random_spins(o.N, 6).astype(np.float32).astype(np.float64)
    kw = dict(solver="heun", dt=1e-3, alpha=0.1, T=T, seed=1, step0=40)
    c = _ctx(g, h)
    n = c.spins(n0)
    c.llg_step(n, 1, **kw)
    assert np.abs(n.double().cpu().numpy()[:, :3] - o.llg(n0, 1, **kw)).max() <= 1e-5
    out = []
    for lean in (1, 0):
        c = _ctx(g, h, lean)
        n = c.spins(n0)
        c.llg_step(n, 5, **kw)
        out.append(n)
    assert (out[0] - out[1]).abs().max().item() <= 2e-6
    assert c.sync_status()[0] == 0


@pytest.mark.parametrize("name", list(CASES))
def test_ragged_columns_and_splits_give_the_same_bits(name):
    g, h = CASES[name]
    n0 = I.random_spins(int(np.prod(g["n_cells"])), 12)
    kw = dict(solver="heun", dt=2e-3, alpha=0.2, T=9.0, seed=4, step0=7)
    out = []
    for o in (dict(), dict(cubic_rows=1), dict(cubic_rows=2), dict(cubic_rows=1, cubic_rows_corr=2),
              dict(planes_per_cta=1), dict(planes_per_cta=3, planes_per_cta_corr=2), dict(planes_per_cta=1000),
              dict(cubic_rows=2, planes_per_cta=3)):
        c = _ctx(g, h, **o)
        n = c.spins(n0)
        c.llg_step(n, 4, **kw)
        out.append(n)
    for n in out[1:]:
        assert torch.equal(n, out[0])


@pytest.mark.parametrize("dims,R", [((30, 30, 30), 12), ((33, 5, 6), 3), ((32, 8, 5), 2)])
def test_replicas_equal_single_calls(dims, R):
    g, h = I.simple_cubic(*dims), SC
    N = int(np.prod(dims))
    temps = [3.0 * r for r in range(R)]
    n0 = np.stack([I.random_spins(N, 40 + r) for r in range(R)])
    kw = dict(solver="heun", dt=1e-3, alpha=0.1, seed=5, step0=5000000000)
    for steps in (3, 40):
        c = _ctx(g, h, **({} if N > 20000 else dict(planes_per_cta=2)))
        x = c.spins(n0)
        c.llg_step_replicas(x, temps, steps, replica=3, **kw)
        for r, T in enumerate(temps):
            y = c.spins(n0[r])
            c.llg_step(y, steps, T=T, replica=3 + r, **kw)
            assert torch.equal(x[r], y), (steps, r)
