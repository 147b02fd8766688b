"""The FP32 passes that hold the loop over a stencil's entries alone: planes of one atom
per cell with neither four nor six bonds (and a crystal, whose passes hold all loops).

One step of every solver against the oracle (the FP32 bound of one step in
test_gpu_lean.py), at every kind of edge; and the bits of a batch of lattices,
whose kernels hold all neighbour loops.
"""
import numpy as np
import pytest

import oracle
from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import inputs as I

pytestmark = pytest.mark.gpu

HEX2 = dict(J=[1.0, 0.1], dmi_kind="interfacial", D=[0.35], K=[0.08], Khat=[[0.1, 0, 1]], B=[0.1, 0, 1.2])
SC2 = dict(J=[1.0, -0.2], dmi_kind="bulk", D=[0.3], K=[0.1], Khat=[[0, 0.2, 1]], B=[0, 0.3, 0.5])
SYSTEMS = {
    "hex_two_shells": (I.hexagonal(33, 17, periodic=(True, True)), HEX2),
    "hex_three_shells_open": (I.hexagonal(9, 31, periodic=(False, True)), dict(HEX2, J=[1.0, 0.1, -0.2])),
    "square_two_shells_open": (I.square(16, 16, periodic=(False, False)), dict(HEX2, J=[1.0, 0.3])),
    "sc_two_shells": (I.simple_cubic(5, 7, 8, periodic=(True, False, True)), SC2),
    "chain_of_two_bonds": (I.square(300, 1, periodic=(True, False)), dict(J=[1.0], B=[0, 0, 1.0])),
}


def _step(c, n, solver, steps=1, **kw):
    c.llg_step(n, steps, solver=solver, dt=1e-3, alpha=0.2, seed=5, step0=3, **kw)
    return n


@pytest.mark.parametrize("name", list(SYSTEMS))
@pytest.mark.parametrize("solver", ["depondt", "heun", "sib", "rk4"])
@pytest.mark.parametrize("T", [0.0, 8.0])
def test_step_matches_oracle(name, solver, T):
    g, h = SYSTEMS[name]
    o, c = oracle.System(g, h), B.Context(g, h, "f32")
    c.set_option("small_path", 0)
    c.set_option("generic_stencil", 1)
    n0 = I.random_spins(o.N, 6).astype(np.float32).astype(np.float64)
    n = _step(c, c.spins(n0), solver, T=T)
    ref = o.llg(n0, 1, solver=solver, dt=1e-3, alpha=0.2, T=T, seed=5, step0=3)
    assert np.abs(n.double().cpu().numpy()[:, :3] - ref).max() <= 1e-5


@pytest.mark.parametrize("solver", ["depondt", "heun", "sib"])
def test_batch_of_lattices_gives_the_bits_of_single_calls(solver):
    systems = [SYSTEMS["hex_two_shells"], (I.hexagonal(20, 15, periodic=(True, False)), dict(HEX2, J=[1.0])),
               SYSTEMS["sc_two_shells"]]
    ctxs = [B.Context(g, h, "f32") for g, h in systems]
    off = np.cumsum([0] + [c.N for c in ctxs])
    n0 = I.random_spins(int(off[-1]), 9)
    x = ctxs[0].spins(n0)
    B.llg_step_batch(ctxs, x, off[:-1].tolist(), [4.0, 0.0, 9.0], 5, solver=solver, dt=1e-3, alpha=0.2, seed=5, step0=3)
    for k, (c, T) in enumerate(zip(ctxs, [4.0, 0.0, 9.0])):
        c.set_option("small_path", 0)
        c.set_option("generic_stencil", 1)
        y = _step(c, c.spins(n0[off[k]:off[k + 1]]), solver, 5, T=T, replica=k)
        assert (x[off[k]:off[k + 1]] == y).all(), k


@pytest.mark.parametrize("name", ["hex_two_shells", "hex_three_shells_open"])
def test_gneb_gives_the_bits_of_the_persistent_kernel_and_of_a_batch(name):
    g, h = SYSTEMS[name]
    M = 6
    ctxs = [B.Context(g, h, "f32"), B.Context(g, h, "f32"), B.Context(g, dict(h, J=[1.0]), "f32")]
    ctxs[1].set_option("gneb_persistent", 1)
    n0 = np.stack([I.perturbed(I.ferromagnet(ctxs[0].N, (0.3 * m, 0.1, 1.0)), 0.2, m) for m in range(M)])
    out = []
    for c in ctxs[:2]:
        x = c.spins(n0)
        v = x * 0
        E, F = c.gneb_step(x, v, n_iter=12, dt=0.05)
        assert c.sync_status()[0] == 0
        out.append((x, v, E, F))
    assert all((a == b).all() for a, b in zip(*out))
    # beside a chain with the unrolled loop
    x = ctxs[0].spins(np.concatenate([n0.reshape(-1, 3)] * 2))
    v = x * 0
    E, F = B.gneb_batch_step([ctxs[0], ctxs[2]], x, v, [0, M * ctxs[0].N], [M, M], n_iter=12, dt=0.05)
    assert (x[:M * ctxs[0].N].reshape(out[0][0].shape) == out[0][0]).all() and (E[:M] == out[0][2]).all()
