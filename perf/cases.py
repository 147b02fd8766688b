"""Measured cases: the calls a program makes of this library, over the sizes it makes them at.

Every case goes through the public binding (``binding.Context`` and the batch functions beside it, ``unet.UNet``).  The
sizes are those of the repository's workloads (``inputs.py``, ``bench.py``) and ragged lattices of the same kinds.
``exact`` restates each method in 64 bits with plain torch, on the lattice as a dense array with rolled neighbours, and
uses nothing of the library.
"""
import math

import numpy as np
import torch

from paper_1901_11350_gb300 import binding as B
from paper_1901_11350_gb300 import unet as UN

MU_B, K_B, GAMMA = 0.05788381806, 0.08617333262, 0.176085963023
C_DIP = 0.0536815112357  # mu_0 / 4 pi in meV A^3 / mu_B^2
CONV = [(32, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (128, 256), (256, 256),
        (384, 128), (128, 128), (192, 64), (64, 64), (96, 32), (32, 32)]  # (cin, cout) of the network's layers
LEVEL = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0]
HEX = [[1, 0, 0], [0.5, math.sqrt(3.0) / 2.0, 0], [0, 0, 1]]
CUBE = [[1, 0, 0], [0, 1, 0], [0, 0, 1]]


# ------------------------------------------------------------------ the cases
def _llg(name, lattice, n, periodic, precision, solver, steps, T, dipole=False, observe=False):
    return dict(name=name, kind="llg", lattice=lattice, n0=n[0], n1=n[1], n2=n[2], p0=periodic[0], p1=periodic[1],
                p2=periodic[2], precision=precision, solver=solver, steps=steps, T=T, dipole=dipole, observe=observe)


def listed():
    return [
        # the paper's small 2D film in full precision: short runs between two looks at energy and torque (an
        # interactive session); bound by launches and latency
        _llg("square32_depondt_f64", "square", (32, 32, 1), (0, 0, 0), "f64", "depondt", 50, 0.0, observe=True),
        # the headline workload: stochastic Heun on a large periodic crystal, three shells and bulk DMI
        _llg("sc128_heun_f32", "sc", (128, 128, 128), (1, 1, 1), "f32", "heun", 50, 10.0),
        # the same physics on a sample whose extents fit no tile, open in one direction
        _llg("sc100x75x50_heun_f32", "sc", (100, 75, 50), (1, 0, 1), "f32", "heun", 50, 10.0),
        # skyrmion dynamics on a large hexagonal monolayer at 5 K
        _llg("hex1024_depondt_f32", "hex", (1024, 1024, 1), (1, 1, 0), "f32", "depondt", 20, 5.0),
        # the same kind of film with the dipole-dipole interaction by FFT
        _llg("hex512_dipole_f32", "hex", (512, 512, 1), (0, 0, 0), "f32", "depondt", 20, 0.0, dipole=True),
        # stochastic-LLG temperature scan: all temperatures of one lattice, the steps between three samples
        dict(name="sllg30_replicas_f32", kind="replicas", L=30, replicas=29, steps=30),
        # Metropolis temperature scan with sampled observables
        dict(name="mc30_f32", kind="mc", L=30, replicas=29, sweeps=16),
        # minimum-energy paths of skyrmion collapse, chains of uneven sizes and image counts stepped together; small
        # steps from the great-circle path, where no image's velocity has been zeroed yet (the sign of v . F decides
        # that, and one rounding can turn it)
        dict(name="gneb12_f32", kind="gneb", chains=12, images_lo=12, images_hi=40, L_lo=64, L_hi=128, iters=20,
             layout=4),
        # relaxation of many random starts together (labels and evaluation of the learned warm start): one short call
        dict(name="vp64_hex128_f32", kind="vp", systems=64, L=128, precision="f32", iters=16),
        # lowest Hessian mode of a skyrmion (one force evaluation of minimum mode following)
        dict(name="lowest_mode_hex128_f64", kind="mode", L=128, krylov=64),
        # the warm-start network: prediction, and loss with gradient, for a batch of lattices
        dict(name="unet_predict_b64", kind="predict", L=128, batch=64),
        dict(name="unet_loss_grad_b64", kind="loss_grad", L=128, batch=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "sc", "sc", "hex", "dipole", "replicas", "mc", "gneb", "vp", "mode", "predict",
                       "loss_grad"])
    bit = lambda: rng.randint(0, 1)  # noqa: E731
    if kind == "small":
        c = _llg("", "square", (_log_int(rng, 8, 64), _log_int(rng, 8, 64), 1), (bit(), bit(), 0),
                 rng.choice(["f64", "f64", "f32"]), rng.choice(["depondt", "heun"]), 50, 0.0, observe=True)
    elif kind == "sc":
        n = tuple(_log_int(rng, 12, 128) for _ in range(3))
        c = _llg("", "sc", n, (bit(), bit(), bit()), "f32", rng.choice(["heun", "heun", "depondt", "sib"]), 50,
                 rng.choice([10.0, 10.0, 0.0]))
    elif kind == "hex":
        c = _llg("", "hex", (_log_int(rng, 64, 1024), _log_int(rng, 64, 1024), 1), (bit(), bit(), 0), "f32",
                 rng.choice(["depondt", "heun"]), 20, rng.choice([5.0, 0.0]))
    elif kind == "dipole":
        c = _llg("", "hex", (_log_int(rng, 48, 512), _log_int(rng, 48, 512), 1), (0, 0, 0), "f32", "depondt", 20,
                 0.0, dipole=True)
    elif kind == "replicas":
        return dict(kind="replicas", L=rng.randint(8, 30), replicas=rng.randint(4, 29), steps=30)
    elif kind == "mc":
        return dict(kind="mc", L=rng.choice([10, 12, 15, 16, 18, 20, 21, 24, 27, 28, 30]),
                    replicas=rng.randint(4, 29), sweeps=16)
    elif kind == "gneb":
        lo, hi = sorted((_log_int(rng, 32, 128), _log_int(rng, 32, 128)))
        m = rng.randint(12, 36)
        return dict(kind="gneb", chains=rng.randint(1, 12), images_lo=m, images_hi=m + rng.randint(0, 4), L_lo=lo,
                    L_hi=hi, iters=20, layout=rng.randint(0, 1 << 20))
    elif kind == "vp":
        return dict(kind="vp", systems=_log_int(rng, 1, 64), L=_log_int(rng, 24, 128),
                    precision=rng.choice(["f32", "f32", "f64"]), iters=16)
    elif kind == "mode":
        return dict(kind="mode", L=_log_int(rng, 24, 128), krylov=rng.randint(16, 64))
    else:
        # every level's pixel count has to be a multiple of 128
        L = rng.choice([64, 96, 128])
        step = {64: 2, 96: 8, 128: 1}[L]
        return dict(kind=kind, L=L, batch=step * rng.randint(1, 64 // step))
    del c["name"]
    return c


# ------------------------------------------------------------------ systems and inputs
def _system(case):
    """Geometry and Hamiltonian of an llg, replicas or mc case."""
    kind = case["kind"]
    if kind in ("replicas", "mc"):
        L = case["L"]
        g = dict(bravais=CUBE, basis=[[0, 0, 0]], n_cells=[L, L, L], periodic=[1, 1, 1], lattice_constant=1.0,
                 mu_s=[2.0])
        return g, dict(B=[0, 0, 0], K=[0.0], Khat=[[0, 0, 1]], J=[1.0])
    n, p = [case["n0"], case["n1"], case["n2"]], [case["p0"], case["p1"], case["p2"]]
    lat = case["lattice"]
    g = dict(bravais=HEX if lat == "hex" else CUBE, basis=[[0, 0, 0]], n_cells=n, periodic=p, lattice_constant=1.0,
             mu_s=[3.0 if case["dipole"] else 2.0])
    if lat == "sc":
        return g, dict(B=[0, 0, 0], K=[0.05], Khat=[[0, 0, 1]], J=[1.0, -0.2, 0.05], dmi_kind="bulk", D=[0.2])
    if lat == "square":
        return g, dict(B=[0, 0, 1.0], K=[0.1], Khat=[[0, 0, 1]], J=[1.0], dmi_kind="interfacial", D=[0.3])
    if case["dipole"]:
        return g, dict(B=[0, 0, 0], K=[0.2], Khat=[[0, 0, 1]], J=[1.0], dmi_kind="interfacial", D=[0.3], dipole="fft")
    return g, dict(B=[0, 0, 1.0], K=[0.07], Khat=[[0, 0, 1]], J=[1.0], dmi_kind="interfacial", D=[0.3])


def _alpha(case):
    return 1.0 if case["kind"] == "replicas" else {"sc": 0.1, "square": 0.3, "hex": 0.5}[case["lattice"]]


def _monolayer(L, D, K, Bz):
    g = dict(bravais=HEX, basis=[[0, 0, 0]], n_cells=[L, L, 1], periodic=[1, 1, 0], lattice_constant=1.0, mu_s=[2.0])
    return g, dict(B=[0, 0, Bz], K=[K], Khat=[[0, 0, 1]], J=[1.0], dmi_kind="interfacial", D=[D])


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _sphere(shape, gen, dtype):
    """Records uniform on the sphere, the pad lane zero."""
    x = torch.randn(tuple(shape) + (3,), generator=gen, device="cuda", dtype=torch.float64)
    return _records(x / x.norm(dim=-1, keepdim=True), dtype)


def _records(x, dtype):
    out = torch.zeros(x.shape[:-1] + (4,), dtype=dtype, device="cuda")
    out[..., :3] = x
    return out


def _dtype(case):
    return torch.float64 if case.get("precision") == "f64" else torch.float32


def _skyrmion(L, radius):
    """Polar and in-plane angle of a Neel skyrmion in the middle of an L x L hexagonal lattice, site order."""
    c1, c0 = torch.meshgrid(torch.arange(L, device="cuda", dtype=torch.float64),
                            torch.arange(L, device="cuda", dtype=torch.float64), indexing="ij")
    x = (c0 + 0.5 * c1 - 0.75 * (L - 1)).reshape(-1)
    y = (HEX[1][1] * (c1 - 0.5 * (L - 1))).reshape(-1)
    r = torch.hypot(x, y)
    return torch.clamp(math.pi * (1 - r / radius), min=0.0), torch.atan2(y, x) + math.pi


def _polar(theta, psi):
    s = torch.sin(theta)
    return torch.stack([s * torch.cos(psi), s * torch.sin(psi), torch.cos(theta)], dim=-1)


def _gneb_layout(case):
    rng = np.random.default_rng(case["layout"])
    return [(int(rng.integers(case["L_lo"], case["L_hi"] + 1)),
             int(rng.integers(case["images_lo"], case["images_hi"] + 1))) for _ in range(case["chains"])]


def _gneb_params(case, seed):
    """(radius, D, K, B) per chain, in the ranges of the collapse workload."""
    rng = np.random.default_rng(int(seed))
    return [(int(rng.integers(5, 9)), float(rng.uniform(0.25, 0.4)), float(rng.uniform(0.05, 0.1)),
             float(rng.uniform(0.5, 2.0))) for _ in range(case["chains"])]


def _vp_params(case, seed):
    rng = np.random.default_rng(int(seed))
    return [(float(rng.uniform(0.1, 0.5)), float(rng.uniform(0.0, 0.2)), float(rng.uniform(0.0, 3.0)))
            for _ in range(case["systems"])]


def _temperatures(case):
    return [10.0 + 14.0 * r / 28.0 for r in range(case["replicas"])]


def _net_params(seed):
    """He-normal weights that BF16 holds exactly (as trained weights are stored), small biases."""
    rng = np.random.default_rng(int(seed))
    parts = []
    for l, (ci, co) in enumerate(CONV):
        w = rng.standard_normal((co, 9, ci)) * math.sqrt(2.0 / (9 * (7 if l == 0 else ci)))
        if l == 0:
            w[:, :, 7:] = 0.0
        w = torch.from_numpy(w).to(torch.bfloat16).float().numpy()
        parts += [w.ravel(), 0.05 * rng.standard_normal(co)]
    parts += [rng.standard_normal(96) / math.sqrt(32.0), 0.1 * rng.standard_normal(3)]
    return np.concatenate(parts).astype(np.float32)


def _net_inputs(case, seed):
    g, n = _gen(seed), case["L"] ** 2
    x = _sphere((case["batch"], n), g, torch.float32)
    f = torch.rand((case["batch"], 4), generator=g, device="cuda")
    f[:, 0] = 1.0
    up = torch.zeros(3, dtype=torch.float64, device="cuda")
    up[2] = 1.0
    t = up + 0.3 * torch.randn((case["batch"], n, 3), generator=g, device="cuda", dtype=torch.float64)
    return x, f, _records(t / t.norm(dim=-1, keepdim=True), torch.float32)


def prepare(case, seed):
    kind, s = case["kind"], dict(case=case)
    if kind == "llg":
        g, h = _system(case)
        s["ctx"] = B.Context(g, h, case["precision"])
        s["n"] = _sphere((s["ctx"].N,), _gen(seed), _dtype(case))
        s["seed"], s["step"] = int(seed) % 100003, 0
    elif kind in ("replicas", "mc"):
        g, h = _system(case)
        s["ctx"] = B.Context(g, h, "f32")
        # partly ordered states, as a scan across the transition meets them
        x = torch.randn((case["replicas"], s["ctx"].N, 3), generator=_gen(seed), device="cuda", dtype=torch.float64)
        x[..., 2] += 1.0
        s["n"] = _records(x / x.norm(dim=-1, keepdim=True), torch.float32)
        s["T"], s["seed"], s["step"] = _temperatures(case), int(seed) % 100003, 0
        if kind == "mc":
            s["cone"] = torch.full((case["replicas"],), 0.7, dtype=torch.float64, device="cuda")
            s["stats"] = torch.zeros((case["replicas"], 8), dtype=torch.float64, device="cuda")
    elif kind == "gneb":
        s["ctxs"], s["offsets"], s["images"], parts, off = [], [], [], [], 0
        for (L, M), (R, D, K, Bz) in zip(_gneb_layout(case), _gneb_params(case, seed)):
            s["ctxs"].append(B.Context(*_monolayer(L, D, K, Bz), "f32"))
            parts.append(_gneb_chain(L, M, R))
            s["offsets"].append(off)
            s["images"].append(M)
            off += M * L * L
        s["start"] = torch.cat(parts)
        s["x"], s["v"] = torch.empty_like(s["start"]), torch.empty_like(s["start"])
    elif kind == "vp":
        L = case["L"]
        s["ctxs"] = [B.Context(*_monolayer(L, *p), case["precision"]) for p in _vp_params(case, seed)]
        s["start"] = _sphere((case["systems"] * L * L,), _gen(seed), _dtype(case))
        s["x"], s["v"] = torch.empty_like(s["start"]), torch.empty_like(s["start"])
        s["offsets"] = [k * L * L for k in range(case["systems"])]
    elif kind == "mode":
        s["ctx"] = B.Context(*_monolayer(case["L"], 0.3, 0.05, 1.5), "f64")
        s["n"], s["start"] = _mode_inputs(case, seed)
        s["mode"] = torch.empty_like(s["start"])
    else:
        s["x"], s["f"], s["t"] = _net_inputs(case, seed)
        s["net"] = UN.UNet(case["L"], case["batch"], _net_params(seed))
        if kind == "predict":
            s["out"] = torch.empty_like(s["x"])
        else:
            s["grad"] = torch.empty(s["net"].n_params, device="cuda")
    return s


def _gneb_chain(L, M, R):
    """The great-circle path from the ferromagnet to the skyrmion."""
    theta, psi = _skyrmion(L, float(R))
    t = torch.linspace(0, 1, M, dtype=torch.float64, device="cuda")[:, None]
    return _records(_polar(theta * t, psi.expand(M, -1)), torch.float32).reshape(-1, 4)


def _mode_inputs(case, seed):
    g = _gen(seed)
    theta, psi = _skyrmion(case["L"], 6.0)
    x = _polar(theta, psi)
    x = x + 0.1 * torch.randn(x.shape, generator=g, device="cuda", dtype=torch.float64)
    v = torch.randn(x.shape, generator=g, device="cuda", dtype=torch.float64)
    return _records(x / x.norm(dim=-1, keepdim=True), torch.float64), _records(v, torch.float64)


# ------------------------------------------------------------------ one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "llg":
        s["ctx"].llg_step(s["n"], case["steps"], solver=case["solver"], dt=1e-3, alpha=_alpha(case), T=case["T"],
                          seed=s["seed"], step0=s["step"])
        s["step"] += case["steps"]
        if not case["observe"]:
            return s["n"]
        e, t = s["ctx"].energy(s["n"]), s["ctx"].max_torque(s["n"])
        # in single precision what is read off is single precision too
        return [s["n"], e, t] if case["precision"] == "f64" else [s["n"], e.float(), t.float()]
    if kind == "replicas":
        s["ctx"].llg_step_replicas(s["n"], s["T"], case["steps"], solver="heun", dt=1e-3, alpha=1.0, seed=s["seed"],
                                   step0=s["step"])
        s["step"] += case["steps"]
        return s["n"]
    if kind == "mc":
        s["ctx"].mc_sweeps(s["n"], s["T"], case["sweeps"], seed=s["seed"], sweep0=s["step"], cone=s["cone"],
                           stats=s["stats"])
        s["step"] += case["sweeps"]
        return [s["n"], s["cone"], s["stats"]]
    if kind == "gneb":
        s["x"].copy_(s["start"])
        s["v"].zero_()
        E, F = B.gneb_batch_step(s["ctxs"], s["x"], s["v"], s["offsets"], s["images"], n_iter=case["iters"], dt=0.02)
        return [s["x"], s["v"], E.float(), F.float()]  # single-precision forces: read off in single precision
    if kind == "vp":
        s["x"].copy_(s["start"])
        s["v"].zero_()
        it, mt = B.minimise_batch(s["ctxs"], s["x"], s["v"], s["offsets"], dt=0.1, tol=1e-6, max_iter=case["iters"],
                                  check_every=256)
        return [s["x"], s["v"], it, mt if case["precision"] == "f64" else mt.astype(np.float32)]
    if kind == "mode":
        s["mode"].copy_(s["start"])
        lam, mode = s["ctx"].lowest_mode(s["n"], s["mode"], case["krylov"])
        # an eigenvector's sign is free: a program that follows a mode turns it towards the one it started from
        return [lam, mode * torch.sign((mode * s["start"]).sum())]
    if kind == "predict":
        return s["net"].predict(s["x"], s["f"], s["out"])
    return [s["net"].loss_grad(s["x"], s["f"], s["t"], s["grad"]), s["grad"]]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Bytes: inputs read once and outputs written once.  Flops: the stencil (6 per exchange bond, 12 more per DMI
    bond, 15 on site), the update of a spin (about 60 per stage, 40 for the thermal field), 2 per multiply-add of a
    convolution, 5 n log2 n per transform."""
    kind = case["kind"]
    if kind in ("llg", "replicas"):
        if kind == "llg":
            n, rec = case["n0"] * case["n1"] * case["n2"], 32 if case["precision"] == "f64" else 16
            bonds = {"sc": 26 * 6 + 6 * 12, "square": 4 * 18, "hex": 6 * 18}[case["lattice"]]
            T, steps = case["T"], case["steps"]
        else:
            n, rec, bonds, T, steps = case["replicas"] * case["L"] ** 3, 16, 36, 1.0, case["steps"]
        per = 2 * (bonds + 15 + 60) + (40 if T > 0 else 0)
        flops = float(n * steps * per)
        if case.get("dipole"):
            P = 4.0 * n
            flops += 2 * steps * (6 * 5 * P * math.log2(P) / 2 + 15 * P)  # three real transforms each way
        return dict(bytes=2.0 * n * rec, flops=flops)
    if kind == "mc":
        n = case["replicas"] * case["L"] ** 3
        return dict(bytes=32.0 * n, flops=float(n * case["sweeps"] * (36 + 90)))
    if kind == "gneb":
        n = sum(M * L * L for L, M in _gneb_layout(case))
        return dict(bytes=64.0 * n, flops=float(n * case["iters"] * (6 * 18 + 15 + 150)))
    if kind == "vp":
        n = case["systems"] * case["L"] ** 2
        rec = 32 if case["precision"] == "f64" else 16
        return dict(bytes=3.0 * n * rec, flops=float(n * case["iters"] * (6 * 18 + 15 + 60)))
    if kind == "mode":
        n, m = case["L"] ** 2, min(case["krylov"], 2 * case["L"] ** 2)
        # per vector the operator, then two orthogonalisations against all earlier vectors (12 flops per spin each)
        return dict(bytes=96.0 * n, flops=float(n * (m * (2 * 6 * 18 + 60) + 12 * m * (m + 1))))
    L, b = case["L"], case["batch"]
    f = sum(2.0 * 9 * ci * co * (L >> lv) ** 2 for (ci, co), lv in zip(CONV, LEVEL)) * b
    npar = sum(co * (9 * ci + 1) for ci, co in CONV) + 99
    if kind == "predict":
        return dict(bytes=b * (32.0 * L * L + 16) + 2.0 * npar, flops=f)
    return dict(bytes=b * (32.0 * L * L + 16) + 6.0 * npar, flops=3 * f)


# ------------------------------------------------------------------ 64-bit restatement
def _bonds(g, h):
    """Directed bonds (offset, J, D vector) of a one-atom lattice, shell by shell."""
    A, offs = np.asarray(g["bravais"], dtype=np.float64), []
    flat = g["n_cells"][2] == 1
    for d in np.ndindex(7, 7, 1 if flat else 7):
        o = (d[0] - 3, d[1] - 3, 0 if flat else d[2] - 3)
        if any(o):
            r = np.asarray(o) @ A
            offs.append((float(np.linalg.norm(r)), o, r))
    lengths = []
    for l, _, _ in sorted(offs, key=lambda x: x[0]):
        if not lengths or l - lengths[-1] > 1e-6:
            lengths.append(l)
    J, D, out = h.get("J", []), h.get("D", []), []
    for l, o, r in offs:
        q = int(np.argmin([abs(l - x) for x in lengths]))
        if q >= max(len(J), len(D)):
            continue
        u = r / l
        e = u if h.get("dmi_kind") == "bulk" else np.array([-u[1], u[0], 0.0])
        out.append((o, J[q] if q < len(J) else 0.0, (D[q] if q < len(D) else 0.0) * e))
    return out


class _Lattice:
    """Fields and energies of states [..., n2, n1, n0, 3] in 64 bits.  D, K, Bz may be tensors over the leading axis."""

    def __init__(self, g, h, scale=None):
        self.nc, self.per = g["n_cells"], g["periodic"]
        self.mu, self.h, self.bonds = g["mu_s"][0], h, _bonds(g, h)
        self.scale = scale  # per system: (D / D of h, K, Bz), each [systems, 1, 1, 1, 1]
        self.kernel = None
        if h.get("dipole"):
            self._dipole_kernel(np.asarray(g["bravais"]))

    def shifted(self, x, o):
        for axis, d, n, p in ((-2, o[0], self.nc[0], self.per[0]), (-3, o[1], self.nc[1], self.per[1]),
                              (-4, o[2], self.nc[2], self.per[2])):
            if d == 0:
                continue
            if not p and abs(d) >= n:
                return torch.zeros_like(x)
            x = torch.roll(x, -d, axis)
            if not p:
                x.narrow(x.dim() + axis, n - d if d > 0 else 0, abs(d)).zero_()
        return x

    def quadratic(self, x):
        """Exchange, DMI and anisotropy field (the part linear in the spins)."""
        out = torch.zeros_like(x)
        for o, J, D in self.bonds:
            y = self.shifted(x, o)
            if J:
                out += J * y
            if np.any(D):
                c = torch.linalg.cross(y, torch.as_tensor(D, device=x.device).expand_as(y))
                out += c if self.scale is None else self.scale[0] * c
        out[..., 2:] += 2 * (self.h["K"][0] if self.scale is None else self.scale[1]) * x[..., 2:]
        if self.kernel is not None:
            out += self._dipole(x)
        return out

    def zeeman(self):
        return self.mu * MU_B * (self.h["B"][2] if self.scale is None else self.scale[2])

    def field(self, x):
        out = self.quadratic(x)
        out[..., 2:] += self.zeeman()
        return out

    def energy(self, x):
        q, dims = self.quadratic(x), (-4, -3, -2, -1)
        z = self.zeeman()
        z = z if not torch.is_tensor(z) else z.reshape(z.shape[0], 1, 1, 1, 1)
        return -(x * q).sum(dims) / 2 - (x[..., 2:] * z).sum(dims)

    def terms(self, x):
        """Total, Zeeman, anisotropy, exchange, DMI, dipole."""
        ez = -float((x[..., 2] * self.zeeman()).sum())
        ea = -self.h["K"][0] * float((x[..., 2] ** 2).sum())
        ex = ed = 0.0
        for o, J, D in self.bonds:
            y = self.shifted(x, o)
            ex -= 0.5 * J * float((x * y).sum())
            ed -= 0.5 * float((x * torch.linalg.cross(y, torch.as_tensor(D, device=x.device).expand_as(y))).sum())
        return torch.tensor([ez + ea + ex + ed, ez, ea, ex, ed, 0.0], dtype=torch.float64)

    def _dipole_kernel(self, A):
        n0, n1 = self.nc[0], self.nc[1]
        d0 = torch.fft.fftfreq(2 * n0, 0.5 / n0, dtype=torch.float64, device="cuda")
        d1 = torch.fft.fftfreq(2 * n1, 0.5 / n1, dtype=torch.float64, device="cuda")
        x = d0[None, :] * A[0, 0] + d1[:, None] * A[1, 0]
        y = d0[None, :] * A[0, 1] + d1[:, None] * A[1, 1]
        r2 = x * x + y * y
        r2[0, 0] = 1.0
        k = torch.stack([3 * x * x / r2 - 1, 3 * x * y / r2, 3 * y * y / r2 - 1, -torch.ones_like(x)]) / r2 ** 1.5
        k[:, 0, 0] = 0.0
        k[:, n1, :] = 0.0
        k[:, :, n0] = 0.0
        self.kernel = torch.fft.rfft2(k)

    def _dipole(self, x):
        n0, n1 = self.nc[0], self.nc[1]
        m = torch.fft.rfft2(self.mu * x[0, 0].permute(2, 0, 1), s=(2 * n1, 2 * n0))
        k = self.kernel
        b = torch.stack([k[0] * m[0] + k[1] * m[1], k[1] * m[0] + k[2] * m[1], k[3] * m[2]])
        b = torch.fft.irfft2(b, s=(2 * n1, 2 * n0))[:, :n1, :n0]
        return (C_DIP * self.mu * b).permute(1, 2, 0)[None, None]


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def _unit(a):
    return a / a.norm(dim=-1, keepdim=True)


def _normals(seed, step, replica, n):
    """Box-Muller normals of Philox4x32-10, counter (site, step, step >> 32, 8 replica), key seed."""
    m32 = 0xFFFFFFFF
    x = [torch.arange(n, device="cuda"), torch.full((n,), step & m32, device="cuda"),
         torch.full((n,), step >> 32, device="cuda"), torch.full((n,), 8 * replica, device="cuda")]
    k0, k1 = seed & m32, seed >> 32
    for r in range(10):
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57  # wraps modulo 2^64: the bits are those of the product
        x = [((p1 >> 32) & m32) ^ x[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ x[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    u = [(v.double() + 0.5) / 4294967296.0 for v in x]
    r0, r1 = torch.sqrt(-2 * torch.log(u[0])), torch.sqrt(-2 * torch.log(u[2]))
    tau = 2 * math.pi
    return torch.stack([r0 * torch.cos(tau * u[1]), r0 * torch.sin(tau * u[1]), r1 * torch.cos(tau * u[3])], -1)


def _rotate(n, A, dt):
    w = A.norm(dim=-1, keepdim=True)
    a = -A / torch.clamp(w, min=1e-300)
    c, s = torch.cos(w * dt), torch.sin(w * dt)
    return n * c + torch.linalg.cross(a, n) * s + a * _dot(a, n) * (1 - c)


def _midpoint(n, A, dt):
    """Solution of x = n + dt (n + x)/2 x A."""
    a = 0.5 * dt * A
    r = n + torch.linalg.cross(n, a)
    return (r + torch.linalg.cross(r, a) + a * _dot(a, r)) / (1 + _dot(a, a))


def _llg_steps(lat, n, solver, dt, alpha, temperatures, seed, steps):
    """n [R, n2, n1, n0, 3], replica r at temperatures[r] on thermal stream r."""
    mu = lat.mu * MU_B
    f = -GAMMA / ((1 + alpha * alpha) * mu)
    A_of = lambda x, b: f * (b + alpha * torch.linalg.cross(x, b))  # noqa: E731
    for step in range(steps):
        th = torch.zeros_like(n)
        for r, T in enumerate(temperatures):
            if T > 0:
                eta = _normals(seed, step, r, n[0].numel() // 3)
                th[r] = math.sqrt(2 * alpha * K_B * T * mu / (GAMMA * dt)) * eta.reshape(n[0].shape)
        A = A_of(n, lat.field(n) + th)
        if solver == "heun":
            k = torch.linalg.cross(n, A)
            p = _unit(n + dt * k)
            n = _unit(n + 0.5 * dt * (k + torch.linalg.cross(p, A_of(p, lat.field(p) + th))))
        elif solver == "depondt":
            p = _rotate(n, A, dt)
            n = _rotate(n, 0.5 * (A + A_of(p, lat.field(p) + th)), dt)
        else:
            p = 0.5 * (n + _midpoint(n, A, dt))
            n = _midpoint(n, A_of(p, lat.field(p) + th), dt)
    return n


def _force(lat, x):
    b = lat.field(x)
    return b - _dot(b, x) * x


def _project_velocity(v, F, dims):
    vf, ff = (v * F).sum(dims, keepdim=True), (F * F).sum(dims, keepdim=True)
    return torch.where((vf > 0) & (ff > 0), vf / ff, torch.zeros_like(vf)) * F


def _exact_vp(case, seed):
    L, S, dt = case["L"], case["systems"], 0.1
    col = lambda k, q=1.0: torch.tensor([p[k] * q for p in _vp_params(case, seed)], dtype=torch.float64,  # noqa: E731
                                        device="cuda").reshape(S, 1, 1, 1, 1)
    lat = _Lattice(*_monolayer(L, 1.0, 0.0, 0.0), scale=(col(0), col(1), col(2)))
    x = _sphere((S * L * L,), _gen(seed), _dtype(case))[:, :3].double().reshape(S, 1, L, L, 3)
    v, F, dims = torch.zeros_like(x), _force(lat, x), (-4, -3, -2, -1)
    for _ in range(case["iters"]):
        x = _unit(x + dt * v + dt * dt / 2 * F)
        G = _force(lat, x)
        v = _project_velocity(v + dt / 2 * (F + G), G, dims)
        F = G
    top = F.norm(dim=-1).amax((-3, -2, -1))
    return [_pad(x.reshape(-1, 3)), _pad(v.reshape(-1, 3)), None, top]


def _gneb_forces(lat, x):
    E, b, M = lat.energy(x), lat.field(x), x.shape[0]
    g = _dot(b, x) * x - b  # gradient, tangent part
    d = x[1:] - x[:-1]
    c = torch.linalg.cross(x[:-1], x[1:]).norm(dim=-1)
    l = (torch.atan2(c, _dot(x[:-1], x[1:])[..., 0]) ** 2).sum((-3, -2, -1)).sqrt()
    e, F = E.tolist(), torch.zeros_like(x)
    top = 1 + int(np.argmax(e[1:-1]))
    for v in range(1, M - 1):
        up, down = e[v + 1] - e[v], e[v] - e[v - 1]
        if up > 0 and down > 0:
            wp, wm = 1.0, 0.0
        elif up < 0 and down < 0:
            wp, wm = 0.0, 1.0
        else:
            hi, lo = max(abs(up), abs(down)), min(abs(up), abs(down))
            wp, wm = (hi, lo) if e[v + 1] > e[v - 1] else (lo, hi)
        t = wp * d[v] + wm * d[v - 1]
        t = t - _dot(t, x[v]) * x[v]
        t = t / t.norm()
        s = (g[v] * t).sum()
        F[v] = -g[v] + (2 * s if v == top else s + 1.0 * (l[v] - l[v - 1])) * t
    return F, E


def _exact_gneb(case, seed):
    xs, vs, Es, Fs, dt = [], [], [], [], 0.02
    for (L, M), (R, D, K, Bz) in zip(_gneb_layout(case), _gneb_params(case, seed)):
        lat = _Lattice(*_monolayer(L, D, K, Bz))
        x = _gneb_chain(L, M, R)[:, :3].double().reshape(M, 1, L, L, 3)
        v = torch.zeros_like(x)
        F, E = _gneb_forces(lat, x)
        for _ in range(case["iters"]):
            y = x.clone()
            y[1:-1] = _unit(x[1:-1] + dt * v[1:-1] + dt * dt / 2 * F[1:-1])
            x = y
            G, E = _gneb_forces(lat, x)
            v = _project_velocity(v + dt / 2 * (F + G), G, (-4, -3, -2, -1))
            F = G
        xs.append(x.reshape(-1, 3))
        vs.append(v.reshape(-1, 3))
        Es.append(E)
        Fs.append(F.norm(dim=-1).max())
    return [_pad(torch.cat(xs)), _pad(torch.cat(vs)), torch.cat(Es), torch.stack(Fs)]


def _exact_mode(case, seed):
    L, m = case["L"], case["krylov"]
    lat = _Lattice(*_monolayer(L, 0.3, 0.05, 1.5))
    n, q = (y[:, :3].reshape(1, 1, L, L, 3) for y in _mode_inputs(case, seed))
    tangent = lambda w: w - _dot(w, n) * n  # noqa: E731
    nB = _dot(n, lat.field(n))
    Q, a, b, start = [], [], [], q.reshape(-1)
    q = tangent(q)
    q = q / q.norm()
    for k in range(m):
        Q.append(q.reshape(-1))
        w = tangent(-lat.quadratic(q)) + nB * q
        a.append(float((w * q).sum()))
        S = torch.stack(Q)
        for _ in range(2):
            w = tangent((w.reshape(-1) - S.T @ (S @ w.reshape(-1))).reshape(n.shape))
        b.append(float(w.norm()))
        q = w / w.norm()
    T = np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1)
    lam, V = np.linalg.eigh(T)
    y = _unit(torch.as_tensor(V[:, 0], device="cuda") @ torch.stack(Q))
    return [float(lam[0]), _pad((y * torch.sign(y @ start)).reshape(-1, 3))]


def _net_forward(params, x, f, L):
    """Network output y [B, L, L, 3] (not normalised)."""
    b = x.shape[0]
    h = torch.cat([x[..., :3].double().reshape(b, L, L, 3), f.double()[:, None, None, :].expand(b, L, L, 4),
                   torch.zeros((b, L, L, 25), dtype=torch.float64, device="cuda")], -1)
    k, skips = 0, {}
    up = lambda z: z.repeat_interleave(2, 1).repeat_interleave(2, 2)  # noqa: E731
    for l, (ci, co) in enumerate(CONV):
        if l in (8, 10, 12):
            h = torch.cat([up(h), skips[{8: 5, 10: 3, 12: 1}[l]]], -1)
        W = params[k:k + co * 9 * ci].reshape(co, 9, ci)
        bias = params[k + co * 9 * ci:k + co * (9 * ci + 1)]
        k += co * (9 * ci + 1)
        z = bias
        for t in range(9):
            z = z + torch.roll(h, (1 - t // 3, 1 - t % 3), (1, 2)) @ W[:, t].T
        h = torch.relu(z)
        if l in (1, 3, 5):
            skips[l] = h
            h = (h[:, ::2, ::2] + h[:, 1::2, ::2] + h[:, ::2, 1::2] + h[:, 1::2, 1::2]) / 4
    return h @ params[k:k + 96].reshape(3, 32).T + params[k + 96:k + 99]


def _exact_net(case, seed):
    L = case["L"]
    x, f, t = _net_inputs(case, seed)
    p = torch.from_numpy(_net_params(seed)).cuda().double()
    grad = case["kind"] == "loss_grad"
    p.requires_grad_(grad)
    out, total, step = [], 0.0, 8
    for c in range(0, case["batch"], step):
        with torch.set_grad_enabled(grad):
            m = _unit(_net_forward(p, x[c:c + step], f[c:c + step], L).reshape(-1, L * L, 3))
            if grad:
                loss = (1 - (m * t[c:c + step, :, :3].double()).sum(-1)).sum() / (case["batch"] * L * L)
                loss.backward()
                total += float(loss)
            else:
                out.append(m)
    return [torch.tensor([total], dtype=torch.float64), p.grad] if grad else _pad(torch.cat(out))


def _pad(x):
    return torch.nn.functional.pad(x, (0, 1))


def exact(case, seed):
    kind = case["kind"]
    if kind == "mc":
        return None  # a decision that falls the other way by one rounding gives another chain
    if kind == "vp":
        return _exact_vp(case, seed)
    if kind == "gneb":
        return _exact_gneb(case, seed)
    if kind == "mode":
        return _exact_mode(case, seed)
    if kind in ("predict", "loss_grad"):
        return _exact_net(case, seed)
    s = prepare(case, seed)
    g, h = _system(case)
    lat, nc = _Lattice(g, h), g["n_cells"]
    n = s["n"][..., :3].double().reshape(-1, nc[2], nc[1], nc[0], 3)
    if kind == "replicas":
        x = _llg_steps(lat, n, "heun", 1e-3, 1.0, s["T"], s["seed"], case["steps"])
        return _pad(x.reshape(case["replicas"], -1, 3))
    x = _llg_steps(lat, n, case["solver"], 1e-3, _alpha(case), [case["T"]], s["seed"], case["steps"])
    if not case["observe"]:
        return _pad(x.reshape(-1, 3))
    return [_pad(x.reshape(-1, 3)), lat.terms(x), torch.linalg.cross(x, lat.field(x)).norm(dim=-1).max().reshape(1)]
