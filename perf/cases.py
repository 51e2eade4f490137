"""Timed cases of the library: the calls that a user's program spends its time
in, from the smallest mesh to the headline one, through the Python front end
(sim.py, guess.py).

Kinds
  step       Sim.step: whole steps of a run (deposit, solve, gather, shrink),
             with the records read back on the device after each group
  batch      Batch.step: independent realisations advancing together
  potential  Sim.solve_potential: one Poisson solve of a given density
  sort       sort_particles: particle order by mesh cell
  pk         power_spectrum: first-order discreteness correction
  pk_jing    power_spectrum_jing: full alias correction
  guess      GuessNet.forward: the network's correction of a residual
  guess_grad GuessNet.loss_grad: one training pair, loss and gradient

All inputs come from the seed: Zel'dovich particles of a power-law spectrum
with the small displacements of an early start for runs, and displaced by
about a cell (clustered, as late snapshots are) where a call takes a snapshot.
"""
import ctypes
import math
import os

import numpy as np
import torch

import paper_1709_04703_gb300 as package
from paper_1709_04703_gb300 import _lib
from paper_1709_04703_gb300.guess import GuessNet
from paper_1709_04703_gb300.sim import (Batch, Sim, power_spectrum, power_spectrum_jing,
                                        sort_particles)

OM, OL = 0.3, 0.7
C_OVER_H0 = 2997.92458


def listed():
    return [
        # the smallest configuration: launches and host round trips decide
        dict(name="step_32", kind="step", n=32, box=250.0, alpha=-2.0, a0=0.02, a1=1.0,
             steps=4000, per_pass=10, rtol=1e-8),
        # the middle configuration, default options
        dict(name="step_128", kind="step", n=128, box=1000.0, alpha=-1.5, a0=0.02, a1=1.0,
             steps=1000, per_pass=10, rtol=1e-7),
        # the headline configuration with the options it is run with
        dict(name="step_256_grouped", kind="step", n=256, box=2000.0, alpha=-1.5, a0=0.01,
             a1=1.0, steps=1000, per_pass=16, rtol=2.4e-4, sort_every=32, inner=4),
        # open boundaries with particles leaving every step, a mesh that is no
        # power of two, the tolerance of the shrinking-against-fixed-box runs
        dict(name="step_192_shrink", kind="step", n=192, box=8192.0, alpha=-1.5, a0=0.30,
             a1=0.38, steps=800, per_pass=10, rtol=1e-5, disp=0.5),
        # the other assignment scheme
        dict(name="step_128_tsc", kind="step", n=128, box=1000.0, alpha=-1.5, a0=0.05, a1=1.0,
             steps=1000, per_pass=10, rtol=1e-5, assignment="tsc"),
        # a suite of small boxes of uneven sizes
        dict(name="batch_12", kind="batch", sizes="32,48,64,96,128,32,64,128,48,96,64,32",
             a0=0.02, a1=1.0, steps=500, per_pass=5, rtol=1e-7),
        # one potential of a given density, open boundaries, from zero
        dict(name="potential_192_open", kind="potential", n=192, bc="open", rtol=1e-7),
        # a ragged number of particles of a clustered snapshot
        dict(name="sort_6m", kind="sort", n_part=6_300_007, n=192),
        # snapshot spectra: every output of a run takes one
        dict(name="pk_256", kind="pk", n_part=16_000_003, n=256, box=2000.0, shot=True),
        dict(name="pk_jing_128", kind="pk_jing", n_part=2_000_003, n=128, box=1000.0),
        # the learned start's forward pass in the open phase, and one training
        # pair of the periodic phase
        dict(name="guess_160", kind="guess", n=160, periodic=False),
        dict(name="guess_grad_96", kind="guess_grad", n=96, periodic=True),
    ]


def _between(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "potential", "sort", "pk", "pk_jing",
                       "guess", "guess_grad"])
    if kind == "step":
        n = rng.choice([32, 48, 64, 96, 128, 192])
        precision = rng.choice(["mixed", "mixed", "fp32"])
        rtol = 2.4e-4 if precision == "fp32" else _between(rng, 1e-8, 1e-4)
        return dict(kind="step", n=n, box=round(rng.uniform(6.0, 10.0) * n, 3), alpha=-1.5,
                    a0=round(rng.uniform(0.02, 0.1), 4), a1=1.0, steps=1000, per_pass=10,
                    rtol=rtol, precision=precision, sort_every=rng.choice([0, 0, 32]),
                    assignment=rng.choice(["cic", "cic", "tsc"]), inner=rng.choice([1, 1, 4]))
    if kind == "batch":
        sizes = [rng.choice([32, 48, 64, 96, 128]) for _ in range(rng.randint(3, 12))]
        return dict(kind="batch", sizes=",".join(map(str, sizes)),
                    a0=round(rng.uniform(0.02, 0.1), 4), a1=1.0, steps=500, per_pass=5,
                    rtol=_between(rng, 1e-8, 1e-6))
    if kind == "potential":
        return dict(kind="potential", n=rng.choice([48, 64, 96, 128, 192, 256]),
                    bc=rng.choice(["open", "periodic"]), rtol=_between(rng, 1e-9, 1e-5))
    if kind == "sort":
        return dict(kind="sort", n_part=int(_between(rng, 3e4, 1.2e7)),
                    n=rng.choice([32, 64, 100, 128, 192, 256, 375]))
    if kind == "pk":
        return dict(kind="pk", n_part=int(_between(rng, 3e4, 1.6e7)),
                    n=rng.choice([32, 64, 96, 125, 128, 192, 256]),
                    box=round(_between(rng, 250.0, 3000.0), 2), shot=rng.random() < 0.5)
    if kind == "pk_jing":
        return dict(kind="pk_jing", n_part=int(_between(rng, 3e4, 4e6)),
                    n=rng.choice([32, 64, 75, 96, 128, 160]),
                    box=round(_between(rng, 250.0, 3000.0), 2))
    if kind == "guess":
        return dict(kind="guess", n=8 * rng.randint(4, 24), periodic=rng.random() < 0.5)
    return dict(kind="guess_grad", n=8 * rng.randint(2, 14), periodic=rng.random() < 0.5)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _generator(seed, stream=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + stream)
    return g


def _wave(n):
    kz = 2 * math.pi * torch.fft.fftfreq(n, device="cuda")
    kx = 2 * math.pi * torch.fft.rfftfreq(n, device="cuda")
    return kx[None, None, :], kz[None, :, None], kz[:, None, None]


def _growth(a):
    """(E(a), dlnD/dlna) of the flat background (growing mode, quadrature)."""
    x = (np.arange(4000) + 0.5) / 4000 * a
    e = math.sqrt(OM / a**3 + OL)
    val = float((x**1.5 / (OM + OL * x**3) ** 1.5).mean() * a)
    return e, -1.5 * OM / (a**3 * e * e) + a / ((a * e) ** 3 * val)


def _lattice(n, alpha, disp, seed, stream=0):
    """Displaced lattice (positions, displacements) in cells, float32 [n^3, 3]."""
    w = torch.fft.rfftn(torch.randn((n, n, n), device="cuda", generator=_generator(seed, stream)))
    kx, ky, kz = _wave(n)
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    dk = w * torch.sqrt(k2 ** (alpha / 2) * torch.exp(-k2 / (2 * (0.5 * math.pi) ** 2)))
    dk[0, 0, 0] = 0
    if n % 2 == 0:  # no Nyquist planes
        dk[n // 2] = 0
        dk[:, n // 2] = 0
        dk[:, :, n // 2] = 0
    psi = torch.stack([torch.fft.irfftn(1j * k * dk / k2, s=(n, n, n)).reshape(-1)
                       for k in (kx, ky, kz)], dim=1)
    psi *= disp / psi.square().sum(dim=1).mean().sqrt()
    g = torch.arange(n, device="cuda", dtype=torch.float32) + 0.5
    Z, Y, X = torch.meshgrid(g, g, g, indexing="ij")
    x = torch.stack([X.reshape(-1), Y.reshape(-1), Z.reshape(-1)], dim=1) + psi
    x = torch.remainder(x, n)
    x[x >= n] = 0.0
    return x, psi


def _ics(n, alpha, disp, a, seed, stream=0):
    """(pos, mom, ids) on the host, as a program that made or read them has."""
    x, psi = _lattice(n, alpha, disp, seed, stream)
    e, f = _growth(a)
    return (x.cpu().numpy(), (psi * (a * a * e * f)).cpu().numpy(),
            np.arange(n**3, dtype=np.int32))


def _snapshot(n_part, n, seed):
    """(pos4, mom4) device records of a clustered snapshot of n_part particles
    on an n^3 mesh, in the order of their lattice."""
    m = 2
    while m**3 < n_part:
        m += 1
    x, psi = _lattice(m, -1.5, 1.5, seed)
    keep = torch.randperm(m**3, device="cuda", generator=_generator(seed, 1))[:n_part]
    keep = keep.sort().values
    x = torch.remainder(x[keep] * (n / m), n)
    x[x >= n] = 0.0
    pos = torch.empty((n_part, 4), device="cuda")
    pos[:, :3] = x
    pos.view(torch.int32)[:, 3] = torch.arange(n_part, device="cuda", dtype=torch.int32)
    mom = torch.zeros((n_part, 4), device="cuda")
    mom[:, :3] = psi[keep]
    return pos, mom


def _density(n, seed):
    """A density contrast (float64) of a clustered box."""
    kx, ky, kz = _wave(n)
    w = torch.fft.rfftn(torch.randn((n, n, n), device="cuda", generator=_generator(seed)))
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    d = torch.fft.irfftn(w * torch.sqrt(k2 ** -0.75 * torch.exp(-k2 / 5.0)), s=(n, n, n))
    d = torch.exp((d - d.mean()) / d.std()).double()
    return d / d.mean() - 1.0


def _pair(n, seed):
    """A start's residual and the correction that removes it (periodic), both
    float32 [1, n, n, n]."""
    kx, ky, kz = _wave(n)
    r = torch.randn((n, n, n), device="cuda", generator=_generator(seed))
    rk = torch.fft.rfftn(r) * torch.exp(-(kx * kx + ky * ky + kz * kz) / 2.0)
    rk[0, 0, 0] = 0
    lam = 2 * (torch.cos(kx) + torch.cos(ky) + torch.cos(kz)) - 6
    lam[0, 0, 0] = 1.0
    r = torch.fft.irfftn(rk, s=(n, n, n))
    e = torch.fft.irfftn(rk / lam, s=(n, n, n))
    c = 1e-3 / r.std()
    return (r * c)[None].contiguous(), (e * c)[None].contiguous()


def _weights():
    """(params, out_scale) of the network that comes with the package."""
    z = np.load(os.path.join(os.path.dirname(package.__file__), "weights",
                             "guess_l4_pm256_10k.npz"))
    return np.asarray(z["params"], np.float32), float(z["out_scale"])


def _boxes(case):
    sizes = [int(v) for v in case["sizes"].split(",")]
    return [(n, 200.0 + 1300.0 * ((0.618 * (i + 1)) % 1.0)) for i, n in enumerate(sizes)]


# --------------------------------------------------------------------------
# state and pass
# --------------------------------------------------------------------------

def _start(state):
    """(Re)start the run of a step or batch state at its first step."""
    case, ics = state["case"], state["ics"]
    if state.get("run") is not None:
        state["run"].close()
    if case["kind"] == "step":
        state["run"] = Sim(*ics, case["n"], case["box"], case["a0"], case["a1"], case["steps"],
                           rtol=case["rtol"], precision=case.get("precision", "mixed"),
                           assignment=case.get("assignment", "cic"),
                           sort_every=case.get("sort_every", 0),
                           inner_vcycles=case.get("inner", 1))
    else:
        state["run"] = Batch(ics, case["a0"], case["a1"], case["steps"], rtol=case["rtol"])
    state["done"] = 0


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case, kind=kind)
    if kind == "step":
        n = case["n"]
        state["ics"] = _ics(n, case["alpha"], case.get("disp", 0.1), case["a0"], seed)
        state["pos4"] = torch.empty((n**3, 4), device="cuda")
        state["mom4"] = torch.empty((n**3, 4), device="cuda")
        _start(state)
    elif kind == "batch":
        state["ics"] = []
        state["out"] = []
        for i, (n, box) in enumerate(_boxes(case)):
            pos, mom, ids = _ics(n, -1.5, 0.1, case["a0"], seed, 1 + i)
            state["ics"].append(dict(pos=pos, mom=mom, ids=ids, n_mesh=n, box=box))
            state["out"].append(tuple(torch.empty((n**3, 4), device="cuda") for _ in range(2)))
        _start(state)
    elif kind == "potential":
        n = case["n"]
        one = (np.full((1, 3), 0.5 * n, np.float32), np.zeros((1, 3), np.float32),
               np.zeros(1, np.int32))
        state["run"] = Sim(*one, n, 1000.0, 0.5, 1.0, 10, rtol=case["rtol"])
        state["delta"] = _density(n, seed)
    elif kind in ("sort", "pk", "pk_jing"):
        state["pos4"], state["mom4"] = _snapshot(case["n_part"], case["n"], seed)
    else:
        params, scale = _weights()
        state["net"] = GuessNet(4, params=params, out_scale=scale)
        state["r"], state["e"] = _pair(case["n"], seed)
    return state


def _records(pos4, mom4, n):
    return {"pos": pos4[:n, :3], "mom": mom4[:n, :3], "id": pos4.view(torch.int32)[:n, 3]}


def run(state):
    case, kind = state["case"], state["kind"]
    if kind in ("step", "batch"):
        if state["done"] + case["per_pass"] > case["steps"]:  # the run is over: the next one
            _start(state)
        state["run"].step(case["per_pass"])
        state["done"] += case["per_pass"]
    if kind == "step":  # the active particles, then those that left, in order
        sim, pos4, mom4 = state["run"], state["pos4"], state["mom4"]
        n = sim.particles_device(pos4, mom4)
        if n < len(pos4):
            _lib.check(_lib.load().pm_get_lightcone(sim._ctx, pos4[n:].data_ptr(),
                                                    mom4[n:].data_ptr(), 0, None))
        return _records(pos4, mom4, len(pos4))
    if kind == "batch":
        b, lib, got = state["run"], _lib.load(), []
        for r, (pos4, mom4) in enumerate(state["out"]):
            n = ctypes.c_int64()
            _lib.check(lib.pm_batch_get_particles(b._b, r, pos4.data_ptr(), mom4.data_ptr(), 0,
                                                  ctypes.byref(n)))
            got.append(_records(pos4, mom4, n.value))
        return got
    if kind == "potential":
        phi, phi64, _, _ = state["run"].solve_potential(state["delta"], 0.5, bc=case["bc"])
        return {"phi": phi, "phi64": phi64}
    if kind == "sort":
        pos, mom = sort_particles(state["pos4"], state["mom4"], case["n"])
        return _records(pos, mom, case["n_part"])
    if kind == "pk":
        k, p, m = power_spectrum(state["pos4"], case["box"], case["n"], case["n"] // 2,
                                 subtract_shot=case["shot"])
        return {"k": k, "P": p, "modes": m}
    if kind == "pk_jing":
        k, p, m, nu, passes = power_spectrum_jing(state["pos4"], case["box"], case["n"],
                                                  case["n"] // 2)
        return {"k": k, "P": p, "modes": m, "slopes": nu, "passes": passes}
    if kind == "guess":
        return state["net"].forward(state["r"], periodic=case["periodic"])
    loss = state["net"].loss_grad(state["r"], state["e"], periodic=case["periodic"])
    return {"loss": loss, "grad": state["net"].grad()}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def work(case):
    """Per step and particle: the records read and written once (64 B), the
    8 (27) weights and the force; per cell: the potential pair of the last
    step read and the new one written (16 B), and one V-cycle."""
    kind = case["kind"]
    if kind in ("step", "batch"):
        sizes = [case["n"]] if kind == "step" else [n for n, _ in _boxes(case)]
        cells = float(sum(n**3 for n in sizes)) * case["per_pass"]
        nodes = 27 if case.get("assignment") == "tsc" else 8
        return {"bytes": (64 + 16) * cells, "flops": (12 * nodes + 80) * cells}
    n = case["n"]
    if kind == "potential":  # about one decimal digit of the residual per V-cycle
        return {"bytes": 20.0 * n**3, "flops": 80.0 * n**3 * -math.log10(case["rtol"])}
    if kind == "sort":
        return {"bytes": 64.0 * case["n_part"], "flops": 0.0}
    if kind in ("pk", "pk_jing"):
        modes = n**3 / 2.0
        alias = 343 * 5 * modes if kind == "pk_jing" else 0.0
        return {"bytes": 16.0 * case["n_part"] + 4.0 * n**3,
                "flops": 2.5 * n**3 * math.log2(n**3) + 10 * modes + alias}
    # 3^3 convolutions 8-8, 8-16, 16-32, 32-64, 96-32, 48-16, 24-8, 8-8 on
    # their levels
    macs = 27 * n**3 * ((64 + 24 * 8 + 64) + (128 + 48 * 16) / 8 + (512 + 96 * 32) / 64
                        + 2048 / 512)
    if kind == "guess":
        return {"bytes": 8.0 * n**3, "flops": 2.0 * macs}
    return {"bytes": 8.0 * n**3, "flops": 6.0 * macs}


# --------------------------------------------------------------------------
# the same results in 64 bits
# --------------------------------------------------------------------------

_GL = np.polynomial.legendre.leggauss(16)


def _tau(a):
    """Conformal time of a, 1/H0: int_0^sqrt(a) 2 du / sqrt(Om + OL u^6)."""
    e = np.linspace(0.0, math.sqrt(a), 65)
    u = 0.5 * (e[1:] + e[:-1])[:, None] + 0.5 * (e[1:] - e[:-1])[:, None] * _GL[0]
    return float((2.0 / np.sqrt(OM + OL * u**6) * _GL[1] * 0.5 * (e[1] - e[0])).sum())


def _a_of_tau(t):
    lo, hi = 1e-9, 4.0
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if _tau(mid) < t else (lo, mid)
    return 0.5 * (lo + hi)


def _axis(u, tsc):
    """First node and the integer weights (2^16 in all) along one axis."""
    q = torch.floor(u.double() * 65536.0).long()
    if tsc:
        i = q >> 16
        f = q & 65535
        w0, w2 = (65536 - f) ** 2 >> 17, f**2 >> 17
        return i - 1, [w0, 65536 - w0 - w2, w2]
    q = q - 32768
    d = q & 65535
    return q >> 16, [65536 - d, d]


def _poisson_periodic(f):
    n = f.shape[0]
    c = torch.cos(2 * math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n)
    lam = 2 * (c[:, None, None] + c[None, :, None] + c[None, None, : n // 2 + 1]) - 6
    lam[0, 0, 0] = 1.0
    fk = torch.fft.rfftn(f) / lam
    fk[0, 0, 0] = 0
    return torch.fft.irfftn(fk, s=f.shape)


def _dst(x, dim):
    """Type-I sine transform along dim: sum_j x_j sin(pi (j+1)(k+1)/(s+1))."""
    s = x.shape[dim]
    z = torch.zeros_like(x.narrow(dim, 0, 1))
    odd = torch.cat([z, x, z, -x.flip(dim)], dim=dim)
    return -0.5 * torch.fft.rfft(odd, dim=dim).imag.narrow(dim, 1, s)


def _poisson_open(f, lo, n):
    """The 7-point solution with the multipole values (to the quadrupole,
    about the box centre) at the ghost centres: the padded potential."""
    s = f.shape[0]
    y = torch.arange(lo - 1, lo + s + 1, device="cuda", dtype=torch.float64) + 0.5 - n / 2
    Z, Y, X = torch.meshgrid(y, y, y, indexing="ij")
    inner = [c[1:-1, 1:-1, 1:-1] for c in (X, Y, Z)]
    r2i = sum(c * c for c in inner)
    r2 = X * X + Y * Y + Z * Z
    q0 = f.sum()
    dip = [(f * c).sum() for c in inner]
    num2 = 0
    for a, ca in enumerate((X, Y, Z)):
        for b, cb in enumerate((X, Y, Z)):
            q = (f * (3 * inner[a] * inner[b] - (r2i if a == b else 0))).sum()
            num2 = num2 + q * ca * cb
    num1 = X * dip[0] + Y * dip[1] + Z * dip[2]
    g = -(q0 / r2.sqrt() + num1 / r2**1.5 + 0.5 * num2 / r2**2.5) / (4 * math.pi)
    rhs = f.clone()
    rhs[0] -= g[0, 1:-1, 1:-1]
    rhs[-1] -= g[-1, 1:-1, 1:-1]
    rhs[:, 0] -= g[1:-1, 0, 1:-1]
    rhs[:, -1] -= g[1:-1, -1, 1:-1]
    rhs[:, :, 0] -= g[1:-1, 1:-1, 0]
    rhs[:, :, -1] -= g[1:-1, 1:-1, -1]
    c = 2 * torch.cos(math.pi * torch.arange(1, s + 1, device="cuda", dtype=torch.float64)
                      / (s + 1)) - 2
    for d in range(3):
        rhs = _dst(rhs, d)
    rhs = rhs / (c[:, None, None] + c[None, :, None] + c[None, None, :])
    for d in range(3):
        rhs = _dst(rhs, d)
    g[1:-1, 1:-1, 1:-1] = rhs * (2.0 / (s + 1)) ** 3
    return g


def _tent(u, tsc):
    """Integral of the assignment's cloud up to u."""
    if not tsc:
        u = np.clip(u, -1.0, 1.0)
        return np.where(u < 0, 0.5 * (u + 1) ** 2, 1 - 0.5 * (1 - u) ** 2)
    v = np.abs(np.clip(u, -1.5, 1.5))
    t = np.where(v < 0.5, 0.5 + 0.75 * v - v**3 / 3, 1 - (1.5 - v) ** 3 / 6)
    return np.where(np.asarray(u) < 0, 1 - t, t)


def _cube(R, n, tsc):
    """(lo, side, periodic) of the active cube."""
    if R > 0.5 * n - 1.0:
        return 0, n, True
    m = math.ceil(R) + (2 if tsc else 1)
    side = min(min(q << j for q in (1, 3, 5, 7) for j in range(12) if q << j >= 2 * m), n)
    return n // 2 - side // 2, side, False


def _cell_order(x, n):
    """Stable order of the mesh cells of the CIC base nodes."""
    c = torch.remainder(torch.floor(x - 0.5).long(), n)
    return torch.sort((c[:, 2] * n + c[:, 1]) * n + c[:, 0], stable=True).indices


def _exact_steps(pos, mom, ids, n, box, case):
    """The first steps of a run: FP64 forces and potentials, records kept in
    float32 as they are stored, so that the same cells are met."""
    tsc = case.get("assignment") == "tsc"
    N0 = len(pos)
    x, p = torch.from_numpy(pos).cuda(), torch.from_numpy(mom).cuda()
    ids = torch.from_numpy(ids).cuda()
    left = []
    da = (case["a1"] - case["a0"]) / case["steps"]
    t1 = _tau(1.0)
    for k in range(case["per_pass"]):
        a, b = case["a0"] + da * k, case["a0"] + da * (k + 1)
        ta, tb = _tau(a), _tau(b)
        dt, ah = tb - ta, _a_of_tau(0.5 * (ta + tb))
        R = [C_OVER_H0 * (t1 - t) / (box / n) + 1.0 for t in (ta, tb)]
        lo, s, per = _cube(R[0], n, tsc)
        if case.get("sort_every", 0) and k % case["sort_every"] == 0:
            order = _cell_order(x, n)
            x, p, ids = x[order], p[order], ids[order]
        x = x + p * np.float32(dt / (2 * a))
        if per:
            x = torch.where(x < 0, x + n, x)
            x = torch.where(x >= n, x - n, x)
        node, wgt = zip(*(_axis(x[:, d], tsc) for d in range(3)))
        m = len(wgt[0])
        ok = torch.ones(len(x), dtype=torch.bool, device="cuda")
        if not per:
            for d in range(3):
                ok &= (node[d] >= lo) & (node[d] + m - 1 <= lo + s - 1)

        def corners():
            for cz in range(m):
                for cy in range(m):
                    for cx in range(m):
                        ix, iy, iz = ((node[d] + c - lo) % (n if per else 1 << 40)
                                      for d, c in enumerate((cx, cy, cz)))
                        yield (iz * s + iy) * s + ix, wgt[0][cx] * wgt[1][cy] * wgt[2][cz]
        rho = torch.zeros(s**3, dtype=torch.int64, device="cuda")
        for at, w in corners():
            rho.index_add_(0, at[ok], w[ok])
        f = rho.double().reshape(s, s, s) / (2.0**48 * N0 / n**3)
        if per:
            f = f - 1.0
        else:
            e = np.arange(lo, lo + s) + 0.5
            w1 = torch.from_numpy(_tent(n / 2 + R[0] - e, tsc)
                                  - _tent(n / 2 - R[0] - e, tsc)).cuda()
            f = f - w1[:, None, None] * w1[None, :, None] * w1[None, None, :]
        f = f * (1.5 * OM / ah)
        if per:
            phi = _poisson_periodic(f)
            grad = [0.5 * (phi.roll(-1, d) - phi.roll(1, d)) for d in (2, 1, 0)]
        else:
            phi = _poisson_open(f, lo, n)
            c = slice(1, -1)
            grad = [0.5 * (phi[c, c, 2:] - phi[c, c, :-2]), 0.5 * (phi[c, 2:, c] - phi[c, :-2, c]),
                    0.5 * (phi[2:, c, c] - phi[:-2, c, c])]
        F = torch.zeros((len(x), 3), dtype=torch.float64, device="cuda")
        for at, w in corners():
            at = torch.where(ok, at, 0)
            for d in range(3):
                F[:, d] += grad[d].reshape(-1)[at] * w
        F = torch.where(ok[:, None], F * 2.0**-48, 0.0)
        p = (p.double() - ah * dt * F).float()
        x = x + p * np.float32(dt / (2 * b))
        if per:
            x = torch.where(x < 0, x + n, x)
            x = torch.where(x >= n, x - n, x)
        if R[1] <= 0.5 * n - 1.0:
            keep = ((x.double() - n / 2).abs() <= R[1]).all(dim=1)
            left.append((x[~keep], p[~keep], ids[~keep]))
            x, p, ids = x[keep], p[keep], ids[keep]
    x, p, ids = (torch.cat(v) for v in zip((x, p, ids), *left))
    return {"pos": x.double(), "mom": p.double(), "id": ids}


def _exact_density(case, seed):
    """The Fourier modes of the snapshot's density, FP64."""
    n = case["n"]
    pos, _ = _snapshot(case["n_part"], n, seed)
    node, wgt = zip(*(_axis(pos[:, d], False) for d in range(3)))
    rho = torch.zeros(n**3, dtype=torch.int64, device="cuda")
    for c in range(8):
        ix, iy, iz = ((node[d] + ((c >> d) & 1)) % n for d in range(3))
        rho.index_add_(0, (iz * n + iy) * n + ix,
                       wgt[0][c & 1] * wgt[1][(c >> 1) & 1] * wgt[2][c >> 2])
    d = rho.double().reshape(n, n, n) / (2.0**48 * case["n_part"] / n**3) - 1.0
    return torch.fft.rfftn(d)


def _exact_pk(case, seed):
    n, box, nb = case["n"], case["box"], case["n"] // 2
    dk = _exact_density(case, seed)
    i = torch.arange(n, device="cuda")
    i = torch.where(i <= n // 2, i, i - n).double()
    ix = torch.arange(n // 2 + 1, device="cuda").double()
    m = torch.sqrt(ix[None, None, :] ** 2 + i[None, :, None] ** 2 + i[:, None, None] ** 2)
    bins = torch.floor(m + 0.5).long() - 1
    sel = (bins >= 0) & (bins < nb)
    wgt = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    wgt[0] = 1.0
    if n % 2 == 0:
        wgt[-1] = 1.0
    wgt = wgt.expand(m.shape)[sel]
    b = bins[sel]
    obs = (dk.real**2 + dk.imag**2)[sel] * (box**3 / float(n) ** 6)
    half = [(math.pi / n) * v.expand(m.shape)[sel]
            for v in (ix[None, None, :], i[None, :, None], i[:, None, None])]

    def binned(v):
        return torch.bincount(b, weights=wgt * v, minlength=nb)
    count = binned(torch.ones_like(obs))
    kmean = binned(m[sel]) * (2 * math.pi / box) / count
    sinc = [torch.where(h == 0, 1.0, torch.sin(h) / torch.where(h == 0, 1.0, h)) for h in half]
    W = (sinc[0] * sinc[1] * sinc[2]) ** 2
    shot = box**3 / case["n_part"] if case.get("shot", True) else 0.0
    P = binned(obs / W**2 - shot) / count
    out = {"k": kmean.cpu().numpy(), "P": P.cpu().numpy(), "modes": count.cpu().numpy()}
    if case["kind"] == "pk":
        return out
    s2 = [torch.sin(h) ** 2 for h in half]
    c1 = torch.ones_like(obs)
    for v in s2:
        c1 = c1 * (1 - 2.0 / 3.0 * v)
    r0 = half[0] ** 2 + half[1] ** 2 + half[2] ** 2

    def slopes(k, p, nu):
        out = nu.copy()
        for q in range(nb):
            lo, hi = max(q - 1, 0), min(q + 1, nb - 1)
            if hi > lo and p[lo] > 0 and p[hi] > 0:
                out[q] = math.log(p[hi] / p[lo]) / math.log(k[hi] / k[lo])
        return np.clip(out, -6.0, 4.0)
    k, p = out["k"], out["P"]
    nu = slopes(k, p, np.full(nb, -1.0))
    passes = 0
    while passes < 30:
        passes += 1
        h = 0.5 * torch.from_numpy(nu).cuda()[b]
        c2 = torch.zeros_like(obs)
        for az in range(-3, 4):
            for ay in range(-3, 4):
                for ax in range(-3, 4):
                    w, r2 = 1.0, 0.0
                    for v, q, al in zip(half, s2, (ax, ay, az)):
                        y = v + math.pi * al
                        zero = y == 0
                        y2 = y * y
                        w = w * torch.where(zero, 1.0, q * q / torch.where(zero, 1.0, y2 * y2))
                        r2 = r2 + y2
                    c2 += w * torch.exp(h * torch.log(r2 / r0))
        p = (binned((obs - shot * c1) / c2) / count).cpu().numpy()
        new = slopes(k, p, nu)
        moved = np.abs(new - nu).max()
        nu = new
        if moved < 1e-6:
            break
    return {"k": k, "P": p, "modes": out["modes"], "slopes": nu, "passes": passes}


def _net64(params, r, scale, periodic):
    """The network in FP64: channels-first fields, the library's parameter
    order (encoder, decoder, output; weights [cout][tap][cin], then biases)."""
    def conv(v, at):
        ci, co = v.shape[1], layers[at][1]
        w = params[offset[at]:offset[at] + 27 * ci * co].reshape(co, 3, 3, 3, ci)
        bias = params[offset[at] + 27 * ci * co:offset[at] + 27 * ci * co + co]
        pad = torch.nn.functional.pad(v, (1,) * 6, mode="circular" if periodic else "constant")
        out = bias.reshape(1, -1, 1, 1, 1).expand(v.shape[0], co, *v.shape[2:])
        for dz in range(3):  # one product per tap: plain matrix products in 64 bits
            for dy in range(3):
                for dx in range(3):
                    sl = pad[:, :, dz:dz + v.shape[2], dy:dy + v.shape[3], dx:dx + v.shape[4]]
                    out = out + torch.einsum("oc,bczyx->bozyx", w[:, dz, dy, dx], sl)
        return out
    layers = [(8, 8), (8, 16), (16, 32), (32, 64), (96, 32), (48, 16), (24, 8), (8, 8)]
    offset = np.cumsum([0] + [27 * ci * co + co for ci, co in layers])
    rms = r.square().mean().sqrt()
    x = torch.cat([(r / rms)[:, None], torch.ones_like(r)[:, None],
                   torch.zeros((1, 6, *r.shape[1:]), dtype=r.dtype, device="cuda")], dim=1)
    e = [torch.relu(conv(x, 0))]
    for l in range(1, 4):
        e.append(torch.relu(conv(torch.nn.functional.avg_pool3d(e[-1], 2), l)))
    d = e[3]
    for q, l in enumerate((2, 1, 0)):
        up = d
        for ax in (2, 3, 4):
            up = up.repeat_interleave(2, dim=ax)
        d = torch.relu(conv(torch.cat([up, e[l]], dim=1), 4 + q))
    return conv(d, 7)[:, 0], rms * scale


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        ics = _ics(case["n"], case["alpha"], case.get("disp", 0.1), case["a0"], seed)
        return _exact_steps(*ics, case["n"], case["box"], case)
    if kind == "batch":
        return [_exact_steps(*_ics(n, -1.5, 0.1, case["a0"], seed, 1 + i), n, box, case)
                for i, (n, box) in enumerate(_boxes(case))]
    if kind == "potential":
        f = _density(case["n"], seed) * (1.5 * OM / 0.5)
        if case["bc"] == "periodic":
            phi = _poisson_periodic(f)
        else:
            phi = _poisson_open(f, 0, case["n"])[1:-1, 1:-1, 1:-1]
        return {"phi": phi, "phi64": phi}
    if kind == "sort":
        pos, mom = _snapshot(case["n_part"], case["n"], seed)
        order = _cell_order(pos[:, :3], case["n"])
        got = _records(pos[order], mom[order], case["n_part"])
        return {"pos": got["pos"].double(), "mom": got["mom"].double(), "id": got["id"]}
    if kind in ("pk", "pk_jing"):
        return _exact_pk(case, seed)
    params, scale = _weights()
    params = torch.from_numpy(params).cuda().double()
    r, e = _pair(case["n"], seed)
    r, e = r.double(), e.double()
    if kind == "guess":
        with torch.no_grad():
            y, s = _net64(params, r, scale, case["periodic"])
        return y * s
    params.requires_grad_(True)
    y, s = _net64(params, r, scale, case["periodic"])
    d = y - e / s
    if case["periodic"]:
        a = sum(d.roll(q, ax) for ax in (1, 2, 3) for q in (-1, 1)) - 6 * d
    else:
        p = torch.nn.functional.pad(d, (1,) * 6)
        c = slice(1, -1)
        a = (p[:, 2:, c, c] + p[:, :-2, c, c] + p[:, c, 2:, c] + p[:, c, :-2, c]
             + p[:, c, c, 2:] + p[:, c, c, :-2] - 6 * d)
    loss = a.square().mean()
    loss.backward()
    return {"loss": float(loss), "grad": params.grad}
