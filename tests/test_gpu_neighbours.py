"""Edges of the shapes the neighbour loop and the relaxation passes are cut into.

* the local field at every kind of edge (extents of one, two and three cells,
  open and periodic directions, several basis atoms, bonds of more than one
  cell, more bonds than one group of six) against the oracle;
* chains on either side of the sizes at which a thread of the GNEB passes takes
  two and four spins, with images that are not whole blocks: one iteration
  against the oracle, the persistent kernel and a batch bit for bit;
* sampled observables of replicas of many blocks.

FP32 bounds: those of the same quantities in test_gpu_parity.py,
test_gpu_relax_fp32.py and test_gpu_replicas.py.
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


def _np(t):
    return t.detach().cpu().numpy()[..., :3].astype(np.float64)


HEX = dict(J=[1.0], dmi_kind="interfacial", D=[0.35], K=[0.08], Khat=[[0.1, 0, 1]], B=[0.1, 0, 1.2])
SC = dict(J=[1.0, -0.2], dmi_kind="bulk", D=[0.3], K=[0.1], Khat=[[0, 0.2, 1]], B=[0, 0.3, 0.5])
TWO = dict(bravais=[[1, 0, 0], [0, 1, 0], [0, 0, 1]], basis=[[0, 0, 0], [0.5, 0.5, 0.5]], lattice_constant=1.0,
           mu_s=[1.0, 2.0])
BCC = dict(J=[1.0, 0.3], K=[0.1, 0.2], Khat=[[0, 0, 1], [1, 0, 0]], B=[0, 0, 1.0])
SYSTEMS = {
    "hex_2x5": (I.hexagonal(2, 5, periodic=(True, False)), HEX),
    "hex_3x3_periodic": (I.hexagonal(3, 3, periodic=(True, True)), HEX),
    "hex_1x40_open": (I.hexagonal(1, 40, periodic=(False, False)), HEX),
    "hex_65x7": (I.hexagonal(65, 7, periodic=(False, True)), HEX),
    "sc_2x3x2": (I.simple_cubic(2, 3, 2), SC),
    "sc_33x2x1_open": (I.simple_cubic(33, 2, 1, periodic=(False, True, False)), SC),
    "sc_5x4x3_open": (I.simple_cubic(5, 4, 3, periodic=(False, False, False)), SC),
    "bcc_3x2x4": (dict(TWO, n_cells=[3, 2, 4], periodic=[1, 0, 1]), BCC),
    "bcc_4x5x3": (dict(TWO, n_cells=[4, 5, 3], periodic=[0, 1, 1]), BCC),
    "square_third_shell": (I.square(7, 6, periodic=(True, False)), dict(J=[1.0, 0.2, -0.3], B=[0, 0, 1.0])),
}


@pytest.mark.parametrize("name", list(SYSTEMS))
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_field_at_every_edge(name, prec):
    g, h = SYSTEMS[name]
    o = oracle.System(g, h)
    c = B.Context(g, h, prec)
    c.set_option("generic_stencil", 1)
    n0 = I.random_spins(o.N, 4).astype(np.float32).astype(np.float64)
    Bo = o.field(n0)
    tol = 1e-12 if prec == "f64" else 1e-5
    assert np.abs(_np(c.effective_field(c.spins(n0))) - Bo).max() <= tol * np.abs(Bo).max()


# spins of a chain around 155648 (two spins per thread) and 311296 (four)
@pytest.mark.parametrize("n0,n1,M", [(97, 89, 18), (97, 89, 19), (129, 101, 23), (129, 101, 24)])
def test_gneb_iteration_of_chains_of_every_block_shape(n0, n1, M):
    g = I.hexagonal(n0, n1, periodic=(True, True), mu_s=2.0)
    h = dict(J=[1.0], dmi_kind="interfacial", D=[0.3], K=[0.07], Khat=[[0, 0, 1]], B=[0, 0, 1.0])
    r = I.site_positions(g)
    ch = I.slerp_chain(I.ferromagnet(I.n_spins(g)), I.neel_skyrmion(r, r.mean(axis=0), 6.0), M, r, r.mean(axis=0))
    ch = ch.astype(np.float32).astype(np.float64)
    o = oracle.System(g, h)
    kw = dict(k_spring=1.0, climbing=True, dt=0.2)
    out = []
    for persistent in (0, 1):
        c = B.Context(g, h, "f32")
        c.set_option("gneb_persistent", persistent)
        x = c.spins(ch)
        v = torch.zeros_like(x)
        E, F = c.gneb_step(x, v, n_iter=1, **kw)
        out.append((x, v, E, F))
    for a, b in zip(*out):
        assert torch.equal(a, b)
    x, v, E, F = out[0]
    xo, vo, Eo, mfo, _ = o.gneb(ch, n_iter=1, **kw)
    assert np.abs(_np(x) - xo).max() <= 1e-5
    assert np.abs(_np(v) - vo).max() <= 1e-5 * max(1.0, np.abs(vo).max())
    assert np.abs(E.cpu().numpy() - Eo).max() <= 1e-8 * np.abs(Eo).max()
    assert abs(F.item() - mfo) <= 1e-5 * mfo
    # in a batch after a small chain
    g2 = I.hexagonal(9, 7, periodic=(True, True), mu_s=2.0)
    c1, c2 = B.Context(g2, h, "f32"), B.Context(g, h, "f32")
    small = I.slerp_chain(I.random_spins(63, 1), I.random_spins(63, 2), 5)
    xb = torch.cat([c1.spins(small).reshape(-1, 4), c2.spins(ch).reshape(-1, 4)])
    vb = torch.zeros_like(xb)
    Eb, Fb = B.gneb_batch_step([c1, c2], xb, vb, [0, 5 * 63], [5, M], n_iter=1, **kw)
    assert torch.equal(xb[5 * 63:], x.reshape(-1, 4)) and torch.equal(vb[5 * 63:], v.reshape(-1, 4))
    assert torch.equal(Eb[5:], E) and Fb[1].item() == F.item()


@pytest.mark.parametrize("L,R", [(7, 1), (13, 5), (30, 3)])
def test_sampled_observables_of_many_blocks(L, R):
    g, h = I.simple_cubic(L, L, L), dict(J=[1.0])
    c = B.Context(g, h, "f32")
    n0 = np.stack([I.random_spins(c.N, 7 + r) for r in range(R)]) + np.array([0, 0, 1.0])
    n0 /= np.linalg.norm(n0, axis=-1, keepdims=True)
    n0 = n0.astype(np.float32).astype(np.float64)
    st = c.sample(c.spins(n0)).cpu().numpy()
    for r in range(R):
        y = n0[r].reshape(L, L, L, 3)
        E = -sum((y * np.roll(y, -1, a)).sum() for a in range(3))
        m = np.linalg.norm(n0[r].sum(axis=0)) / c.N
        want = np.array([m, m * m, m ** 4, E, E * E, 1, 0, 0])
        assert np.all(np.abs(st[r] - want) <= 1e-6 * np.abs(want) * np.array([1, 2, 4, 1, 2, 0, 0, 0]))


@pytest.mark.parametrize("tilt", [0.0, 0.4])
@pytest.mark.parametrize("n0,n1", [(257, 512), (400, 301)])
def test_dipole_columns_of_films_in_and_out_of_the_plane(tilt, n0, n1):
    # a film in the xy plane has no xz and yz components, a tilted one all six
    # (the bound of the direct sum in test_gpu_parity.py)
    g = I.hexagonal(n0, n1, mu_s=3.0)
    g = dict(g, bravais=[g["bravais"][0], [g["bravais"][1][0], g["bravais"][1][1], tilt], g["bravais"][2]])
    n = I.random_spins(n0 * n1, 13)
    c = B.Context(g, dict(J=[1.0], dipole="fft"), "f32")
    Bf = _np(c.effective_field(c.spins(n)))
    o = oracle.System(g, dict(J=[1.0], dipole="direct"))
    idx = np.concatenate([np.random.default_rng(1).choice(o.N, 60, replace=False), [0, n0 - 1, o.N - 1]])
    ref = o.field(n, dipole="none")[idx] + o.dipole_field_direct_at(n, idx)
    assert np.abs(Bf[idx] - ref).max() <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("n0,n1", [(512, 512), (300, 283)])
def test_steps_with_dipoles_are_the_same_in_every_run(n0, n1):
    # every pass is launched to run beside the end of the one before it: what
    # that one writes must not be read before it has ended
    g = I.hexagonal(n0, n1, mu_s=3.0)
    c = B.Context(g, dict(J=[1.0], K=[0.2], Khat=[[0, 0, 1]], dmi_kind="interfacial", D=[0.3], dipole="fft"), "f32")
    n = I.random_spins(n0 * n1, 3)
    out = []
    for generic in (0, 0, 0, 0, 1):
        c.set_option("generic_fft", generic)
        x = c.spins(n)
        torch.cuda.synchronize()
        c.llg_step(x, 20, solver="depondt", dt=1e-3, alpha=0.5)
        out.append(x)
    for x in out[1:4]:
        assert torch.equal(x, out[0])
    # 40 evaluations whose fields differ by 2e-6 (test_gpu_parity.py) turn a spin
    # by a hundredth of a radian each
    assert (out[4] - out[0]).abs().max().item() <= 1e-5
