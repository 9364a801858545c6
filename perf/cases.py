"""The work that users of this framework have it do, as measurable cases.

A 2D pass advances a batch of members by the steps between two diagnostic
events, runs the sub-volume balance of the new time and reads the state (the
moments, or the populations as a checkpoint holds them).  A 3D pass does the
same without the state (the 3D handle gives it to the host only).  An adjoint
pass is one evaluation of the differentiable objective with its gradients.

What an FP32 handle computes is kept as float32 (its populations, its
statistics), what an FP64 handle computes as float64.
"""
import math
import random

import numpy as np
import torch

import paper_1809_06735_gb300 as lbm
from paper_1809_06735_gb300 import adjoint

DEV = "cuda"


def _ints(text):
    return [int(v) for v in str(text).split(",")]


def _floats(text):
    return [float(v) for v in str(text).split(",")]


def _d2(name=None, grids="512x512", per_grid=1, precision=32, taus="0.52", force=0, kf=4,
        u=0.02, alpha=0.0, F0=0.0, FR0=0.0, collision=0, Cs=0.0, steps=100, sizes="4,16,64",
        boxes="all", graph=0, state="populations", hist=False, start="random_phase", kpeak=8):
    case = dict(locals())
    if name is None:
        del case["name"]
    return {"kind": "d2", **case}


def _d3(name=None, nx=64, ny=64, nz=64, members=1, lattice=19, precision=32, terms=64,
        tau=0.52, force=0, kf=1, u=0.02, alpha=0.0, steps=20, sizes="4,16", boxes=0):
    case = dict(locals())
    if name is None:
        del case["name"]
    return {"kind": "d3", **case}


def _adjoint(name=None, nx=256, ny=256, tau=0.55, kf=4, alpha=1e-4, u=0.03, L=16, n0=1000,
             n1=2000, every=100, precision=64):
    case = dict(locals())
    if name is None:
        del case["name"]
    return {"kind": "adjoint", **case}


def listed():
    return [
        # the plain method at its smallest: one FP64 Taylor-Green member, an
        # event every 100 steps; launches and latency
        _d2("taylor_green_64_fp64", "64x64", 1, 64, "0.6", steps=100, sizes="4,8,16,32",
            state="moments", start="taylor_green"),
        # one plain FP64 run of ordinary size under the Kolmogorov force
        _d2("plain_512_fp64", "512x512", 1, 64, "0.52", force=1, u=0.03, alpha=1e-4, steps=100,
            sizes="2,4,8,16,32,64,128,256", state="moments"),
        # the decaying ensemble: 64 seeds, random boxes inside the domain
        _d2("decaying_64x512_fp32", "512x512", 64, 32, "0.52", steps=200,
            sizes="2,4,8,16,32,64,128,256", boxes="table1", graph=98, kpeak=16),
        # the forced tau sweep: uneven grids in one batch, every origin
        _d2("tau_sweep_15_uneven_fp32", "256x256,512x512,1024x1024", 1, 32,
            "0.505,0.51,0.52,0.55,0.6", force=1, u=0.03, alpha=1e-4, steps=200,
            sizes="2,4,8,16,32,64,128,256,512", graph=98, kpeak=16),
        # the largest single run, every origin of every size
        _d2("large_8192_fp32", "8192x8192", 1, 32, "0.51", force=1, u=0.03, alpha=1e-5,
            steps=100, sizes="2,4,8,16,32,64,128,256,512,1024,2048,4096", graph=98,
            state="moments", kpeak=128),
        # turbulence under the shell force and large-scale damping (the
        # trend's amplitudes), the sizes of its error statistics
        _d2("paper_forcing_64x256_fp32", "256x256", 64, 32, "0.52", force=2, F0=2e-5, FR0=1e-2,
            u=0.01, steps=100, sizes="3,13,51,128,181", graph=50),
        # the two variable-viscosity collisions that ensembles are run with
        _d2("smagorinsky_16x512_fp32", "512x512", 16, 32, "0.51", collision=1, Cs=0.1, steps=100,
            sizes="4,16,64", boxes="table1", graph=20),
        _d2("entropic_16x512_fp32", "512x512", 16, 32, "0.51", collision=3, steps=100,
            sizes="4,16,64", boxes="table1", graph=20),
        # grids that no vector width divides, with the error distributions
        _d2("ragged_6x_fp32", "251x187,509x383", 3, 32, "0.53,0.56", force=1, u=0.03, alpha=1e-4,
            steps=50, sizes="3,10,40,100", hist=True),
        # gradients of the box-averaged dissipation, forward and reverse
        _adjoint("adjoint_256_fp64"),
        # three dimensions: D3Q19 stepping of a batch with FP32 terms over
        # random boxes, and D3Q27 with FP64 terms over every origin
        _d3("d3q19_2x128_fp32", 128, 128, 128, 2, 19, 32, 32, tau=0.52, force=1, alpha=1e-4,
            steps=100, sizes="4,8,16,32,64", boxes=20000),
        _d3("d3q27_64_fp32", 64, 64, 64, 1, 27, 32, 64, tau=0.53, steps=50, sizes="2,4,8,16,32,64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _some_sizes(rng, n, most):
    got = {max(1, min(n, _log(rng, 2, n))) for _ in range(rng.randint(3, most))}
    return ",".join(str(v) for v in sorted(got))


def draw(rng):
    kind = rng.choice(["small64", "plain64", "ensemble", "ensemble", "sweep", "large", "paper",
                       "collision", "ragged", "adjoint", "d3", "d3"])
    if kind in ("small64", "plain64"):
        n = _log(rng, 24, 160) if kind == "small64" else _log(rng, 160, 1024)
        ny = max(20, int(n * rng.uniform(0.6, 1.4)))
        return _d2(None, "%dx%d" % (n, ny), rng.randint(1, 3), 64, "%.3f" % rng.uniform(0.515, 0.7),
                   force=rng.randint(0, 1), u=0.03, alpha=1e-4, steps=rng.randint(20, 150),
                   sizes=_some_sizes(rng, min(n, ny), 6), state="moments")
    if kind == "ensemble":
        nx, ny = 4 * _log(rng, 16, 256), _log(rng, 64, 1024)
        most = max(1, (1 << 24) // (nx * ny))
        return _d2(None, "%dx%d" % (nx, ny), min(96, _log(rng, 1, most)), 32,
                   "%.3f" % rng.uniform(0.51, 0.6), force=rng.randint(0, 1), u=0.03, alpha=1e-4,
                   steps=rng.randint(30, 200), sizes=_some_sizes(rng, min(nx, ny) // 2, 8),
                   boxes=rng.choice(["table1", "all"]), graph=rng.choice([0, 20, 98]),
                   kpeak=max(8, max(nx, ny) // 32))
    if kind == "sweep":
        grids = ",".join("%dx%d" % (4 * _log(rng, 16, 256), _log(rng, 64, 1024))
                         for _ in range(rng.randint(2, 3)))
        taus = ",".join("%.3f" % rng.uniform(0.51, 0.7) for _ in range(rng.randint(2, 4)))
        return _d2(None, grids, 1, 32, taus, force=1, u=0.03, alpha=1e-4,
                   steps=rng.randint(30, 200), sizes=_some_sizes(rng, 512, 8), graph=50,
                   kpeak=16)
    if kind == "large":
        nx, ny = 4 * _log(rng, 512, 1792), _log(rng, 2048, 7168)
        return _d2(None, "%dx%d" % (nx, ny), 1, 32, "0.51", force=1, u=0.03, alpha=1e-5,
                   steps=rng.randint(20, 100), sizes=_some_sizes(rng, min(nx, ny) // 2, 10),
                   graph=rng.choice([0, 50]), state="moments", kpeak=max(nx, ny) // 64)
    if kind == "paper":
        n = 4 * _log(rng, 32, 96)
        return _d2(None, "%dx%d" % (n, n), _log(rng, 4, 64), rng.choice([32, 32, 32, 64]),
                   "%.3f" % rng.uniform(0.515, 0.6), force=2, F0=2e-5, FR0=1e-2, u=0.01,
                   steps=rng.randint(20, 60), sizes=_some_sizes(rng, n, 5), graph=rng.choice([0, 20]))
    if kind == "collision":
        nx, ny = 4 * _log(rng, 32, 192), _log(rng, 128, 768)
        return _d2(None, "%dx%d" % (nx, ny), _log(rng, 2, 24), 32, "%.3f" % rng.uniform(0.505, 0.55),
                   collision=rng.randint(1, 3), Cs=0.1, force=rng.randint(0, 1), u=0.02,
                   steps=rng.randint(20, 100), sizes=_some_sizes(rng, min(nx, ny) // 2, 4),
                   boxes="table1", graph=rng.choice([0, 20]))
    if kind == "ragged":
        grids = ",".join("%dx%d" % (4 * _log(rng, 12, 160) + rng.randint(1, 3), _log(rng, 37, 700))
                         for _ in range(rng.randint(1, 3)))
        return _d2(None, grids, rng.randint(1, 3), 32, "%.3f" % rng.uniform(0.52, 0.6), force=1,
                   u=0.03, alpha=1e-4, steps=rng.randint(20, 80), sizes=_some_sizes(rng, 100, 5),
                   hist=bool(rng.randint(0, 1)))
    if kind == "adjoint":
        nx, ny = _log(rng, 40, 320), _log(rng, 40, 320)
        n1 = _log(rng, 100, 1000)
        return _adjoint(None, nx, ny, round(rng.uniform(0.53, 0.6), 3), 4, 1e-4, 0.03,
                        rng.randint(4, 36), n1 // 2, n1, rng.choice([50, 100]),
                        rng.choice([64, 64, 32]))
    prec = rng.choice([32, 32, 64])
    nx = 4 * _log(rng, 6, 32) + rng.choice([0, 0, 0, 1, 2])
    ny, nz = _log(rng, 20, 128), _log(rng, 20, 128)
    return _d3(None, nx, ny, nz, rng.randint(1, 3), rng.choice([19, 27]), prec,
               32 if prec == 32 and rng.random() < 0.5 else 64, round(rng.uniform(0.51, 0.6), 3),
               rng.randint(0, 1), 1, 0.02, 1e-4, rng.randint(10, 100),
               _some_sizes(rng, min(nx, ny, nz), 6), rng.choice([0, 0, 5000]))


# ---------------------------------------------------------------------------
# What a case's members are, and their initial fields (on the GPU, FP64)
# ---------------------------------------------------------------------------

def _laminar_F0(n, tau, kf, alpha, u):
    nu, k = (tau - 0.5) / 3.0, 2.0 * math.pi * kf / n
    return u * (nu * k * k + alpha)


def _groups(c):
    """Members of equal grids: [(nx, ny, [tau], [F0])], in the handle's order."""
    out = []
    for g in c["grids"].split(","):
        nx, ny = (int(v) for v in g.split("x"))
        taus = [t for t in _floats(c["taus"]) for _ in range(c["per_grid"])]
        F0 = [_laminar_F0(max(nx, ny), t, c["kf"], c["alpha"], c["u"]) if c["force"] == 1 else c["F0"]
              for t in taus]
        out.append((nx, ny, taus, F0))
    return out


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _wave(nx, ny):
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, dtype=torch.float64, device=DEV)
    ky = torch.fft.fftfreq(ny, 1.0 / ny, dtype=torch.float64, device=DEV)[:, None]
    return kx, ky, 2.0 * math.pi * kx / nx, 2.0 * math.pi * ky / ny


def _random_phase(nx, ny, gen, u_rms, kpeak=8):
    """Incompressible random-phase flow with E(k) ~ k^4 exp(-2 (k/kpeak)^2)
    and its zero-Mach density, as decaying turbulence is started."""
    kx, ky, wx, wy = _wave(nx, ny)
    k = torch.sqrt(kx ** 2 + ky ** 2)
    th = 2.0 * math.pi * torch.rand(k.shape, generator=gen, dtype=torch.float64, device=DEV)
    amp = torch.sqrt(torch.exp(-2.0 * (k / kpeak) ** 2) * k)
    amp[(k == 0) | (2 * kx.abs() == nx) | (2 * ky.abs() == ny)] = 0.0
    ph = torch.polar(amp, th)
    inv = lambda a: torch.fft.irfft2(a, s=(ny, nx))  # noqa: E731
    ph = torch.fft.rfft2(inv(ph))
    ux, uy = inv(1j * wy * ph), inv(-1j * wx * ph)
    s = u_rms / torch.sqrt((ux ** 2 + uy ** 2).mean())
    ux, uy, ph = ux * s, uy * s, ph * s
    xx, xy, yy = inv(-wx * wy * ph), inv(-wy * wy * ph), inv(wx * wx * ph)  # d_x u, d_y u, d_x v
    src = torch.fft.rfft2(-(2.0 * xx * xx + 2.0 * xy * yy))
    k2 = wx ** 2 + wy ** 2
    k2[0, 0] = 1.0
    src[0, 0] = 0.0
    return 1.0 + 3.0 * inv(-src / k2), ux, uy


def _taylor_green(nx, ny, gen, u0=0.01):
    a = torch.rand(3, generator=gen, dtype=torch.float64, device=DEV)
    u0 = u0 * (0.8 + 0.4 * a[2])
    x = 2.0 * math.pi * (torch.arange(nx, dtype=torch.float64, device=DEV) / nx + a[0])
    y = 2.0 * math.pi * (torch.arange(ny, dtype=torch.float64, device=DEV)[:, None] / ny + a[1])
    p = -0.25 * u0 * u0 * (torch.cos(2 * x) + torch.cos(2 * y))
    return 1.0 + 3.0 * p, u0 * torch.sin(x) * torch.cos(y), -u0 * torch.cos(x) * torch.sin(y)


def _fields(c, seed):
    """Per group of equal grids: rho, u_x, u_y, each [members, ny, nx]."""
    gen, out = _gen(seed), []
    for nx, ny, taus, _ in _groups(c):
        make = _taylor_green if c["start"] == "taylor_green" else lambda *a: _random_phase(*a, c["u"], c["kpeak"])
        got = [make(nx, ny, gen) for _ in taus]
        out.append(tuple(torch.stack([f[q] for f in got]) for q in range(3)))
    return out


def _fields3(c, seed):
    """rho, u of every member, [members][4][nz, ny, nx]: a few Fourier modes."""
    gen, out = _gen(seed), []
    ax = [2.0 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n
          for n in (c["nx"], c["ny"], c["nz"])]
    x, y, z = ax[0], ax[1][:, None], ax[2][:, None, None]
    for _ in range(c["members"]):
        f = []
        for q in range(4):
            r = torch.rand(6, 5, generator=gen, dtype=torch.float64, device=DEV).cpu()
            a = sum((float(m[4]) - 0.4) * torch.cos(int(4 * m[0]) * x + int(4 * m[1]) * y +
                                                    int(1 + 3 * m[2]) * z + 6.28 * float(m[3])) for m in r)
            f.append((1.0 if q == 0 else 0.0) + (0.02 * c["u"] if q == 0 else 0.5 * c["u"]) * a)
        out.append(f)
    return out


def _origins(c, seed, n, dim=2):
    """Random boxes inside the domain: one list per size, or None for all."""
    if c["boxes"] in ("all", 0):
        return None
    g = np.random.default_rng(int(seed) & 0x7FFFFFFF)
    out = []
    for L in _ints(c["sizes"]):
        if c["boxes"] == "table1":  # the paper's counts, scaled with the grid
            s = n / 256.0
            count = 1 if L >= n else 1000 if L >= 100 * s else 5000 if L >= 10 * s else 10000
        else:
            count = int(c["boxes"])
        out.append(g.integers(0, max(1, n - L + 1), size=(count, dim)).astype(np.int32))
    return out


DELTA_EDGES = np.linspace(0.0, 0.5, 65)
MACH_EDGES = np.linspace(0.0, 0.2, 65)


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = c = case
    if c["kind"] == "d2":
        groups = _groups(c)
        s.members = [lbm.Member(nx, ny, t, 1.0, c["force"], c["kf"], F0, c["alpha"], 0.0, c["FR0"],
                                c["collision"], c["Cs"])
                     for nx, ny, taus, F0s in groups for t, F0 in zip(taus, F0s)]
        s.lat = lbm.Lattice(s.members, precision=c["precision"], diag_every=c["steps"],
                            graph_steps=c["graph"])
        m = 0
        for f in _fields(c, seed):
            n = f[0].shape[0]
            s.lat.init_fields_batch(list(range(m, m + n)), *f)
            m += n
        s.every, s.Ls = list(range(len(s.members))), _ints(c["sizes"])
        s.boxes = _origins(c, seed, min(min(nx, ny) for nx, ny, _, _ in groups))
        s.dtype = torch.float32 if c["precision"] == 32 else torch.float64
        if c["state"] == "populations":  # the checkpoint's buffers, one per grid
            s.out = [torch.empty(len(t), 9, ny, nx, dtype=torch.float64, device=DEV)
                     for nx, ny, t, _ in groups]
    elif c["kind"] == "d3":
        s.lat = lbm.Lattice3D([lbm.Member3(c["nx"], c["ny"], c["nz"], c["tau"], 1.0, c["force"], c["kf"],
                                           _F0_3(c), c["alpha"])] * c["members"],
                              precision=c["precision"], diag_every=c["steps"], lattice=c["lattice"],
                              diag_precision=c["terms"])
        for m, f in enumerate(_fields3(c, seed)):
            s.lat.init_fields(m, *[a.cpu().numpy() for a in f])
        s.Ls = _ints(c["sizes"])
        s.boxes = _origins(c, seed, min(c["nx"], c["ny"], c["nz"]), 3)
    else:
        s.spec = adjoint.ObjectiveSpec(c["nx"], c["ny"], c["kf"], c["alpha"], c["n0"], c["n1"], (0, 0),
                                       c["L"], c["precision"], c["every"])
        s.f0 = _adjoint_f0(c, seed).requires_grad_()
        s.tau = torch.tensor(c["tau"], dtype=torch.float64, requires_grad=True)
        s.F0 = torch.tensor(_laminar_F0(max(c["nx"], c["ny"]), c["tau"], c["kf"], c["alpha"], c["u"]),
                            dtype=torch.float64, requires_grad=True)
    return s


def _F0_3(c):
    return _laminar_F0(max(c["nx"], c["ny"], c["nz"]), c["tau"], c["kf"], c["alpha"], c["u"]) if c["force"] else 0.0


def _kept(a, precision):
    return a.astype(np.float32) if precision == 32 else a


def run(s):
    c, out = s.case, {}
    if c["kind"] == "d2":
        s.lat.step(c["steps"])
        if c["hist"]:
            got = s.lat.subvolume_distributions(s.every, s.Ls, DELTA_EDGES, MACH_EDGES, s.boxes)
            out["delta_hist"], out["mach_hist"] = got["delta_hist"], got["mach_hist"]
            out["mach"], stats = _kept(got["mach"], c["precision"]), got["stats"]
        else:
            stats = s.lat.subvolume_balance_batch(s.every, s.Ls, s.boxes)
        out["stats"] = _kept(stats, c["precision"])
        if c["state"] == "moments":
            out["state"] = [{k: v.to(s.dtype) for k, v in s.lat.moments(m).items()} for m in s.every]
        else:
            m = 0
            for buf in s.out:
                for f in buf:
                    s.lat.get_populations(m, out=f)
                    m += 1
            out["state"] = [buf.to(s.dtype) for buf in s.out]
    elif c["kind"] == "d3":
        s.lat.step(c["steps"])
        got = [s.lat.subvolume_balance(m, s.Ls, s.boxes, per_box=True) for m in range(c["members"])]
        out["boxes"] = [b.to(torch.float32) if c["precision"] == 32 else b for _, b in got]
        out["stats"] = _kept(np.stack([st for st, _ in got]), c["precision"])
    else:
        s.f0.grad = s.tau.grad = s.F0.grad = None
        J = adjoint.box_dissipation(s.tau, s.F0, s.f0, s.spec)
        J.backward()
        got = {"J": J.detach(), "dtau": s.tau.grad, "dF0": s.F0.grad, "df0": s.f0.grad}
        out = {k: v.to(torch.float32) if c["precision"] == 32 else v for k, v in got.items()}
    return out


def work(case):
    """One pass's inputs read once and outputs written once (the state as the
    handle stores it), and the arithmetic of its steps and term fields."""
    c = case
    if c["kind"] == "adjoint":
        cells, steps = c["nx"] * c["ny"], c["n1"]
        return {"bytes": 2 * 72.0 * cells, "flops": (148 + 148 + 206.0) * cells * steps}
    es, bytes_, flops = c["precision"] // 8, 0.0, 0.0
    if c["kind"] == "d3":
        q, cells = c["lattice"], c["members"] * c["nx"] * c["ny"] * c["nz"]
        rows = c["members"] * len(_ints(c["sizes"])) * (c["boxes"] or cells // c["members"])
        return {"bytes": 2.0 * q * es * cells + 15 * 8.0 * rows,
                "flops": 18.0 * q * cells * c["steps"] + 800.0 * cells}
    for nx, ny, taus, _ in _groups(c):
        cells = nx * ny * len(taus)
        read = 4 * es if c["state"] == "moments" else 9 * es
        bytes_ += (2 * 9 * es + read) * cells
        flops += (150.0 * c["steps"] + 400.0) * cells
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
C3 = [(x, y, z) for x in (0, 1, -1) for y in (0, 1, -1) for z in (0, 1, -1)]


def _lattice(q):
    """Velocities and weights; only D2Q9's order is a matter of outputs."""
    if q == 9:
        return C2, W2
    cs = [c for c in C3 if q == 27 or sum(map(abs, c)) < 3]
    w = {0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216} if q == 27 else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
    return cs, [w[sum(map(abs, c))] for c in cs]


def _dot(c, a):
    """c . a over the axes where c is not 0; None for none."""
    s = None
    for ci, ai in zip(c, a):
        if ci:
            t = ai if ci > 0 else -ai
            s = t if s is None else s + t
    return s


def _moments(f, cs):
    rho = sum(f[1:], f[0])
    return rho, [sum(ci[a] * fi for ci, fi in zip(cs, f) if ci[a]) for a in range(len(cs[0]))]


def _feq(rho, u, c, w):
    cu, uu = _dot(c, u), sum(a * a for a in u)
    base = 1.0 - 1.5 * uu
    return w * rho * (base if cu is None else base + cu * (3.0 + 4.5 * cu))


def _entropic_feq(rho, u, c, w):
    p = w * rho
    for ci, a in zip(c, u):
        s = torch.sqrt(1.0 + 3.0 * a * a)
        p = p * (2.0 - s) * ((2.0 * a + s) / (1.0 - a)) ** ci
    return p


def _entropy_root(f, d):
    """alpha > 1 with H(f + alpha d) = H(f), by Newton from 2 on
    g = sum f phi(a y) - a sum d ln(1 + y), y = d/f, phi(z) = (1 + z) ln(1 + z) - z."""
    y = [di / fi for di, fi in zip(d, f)]
    s2 = sum(di * torch.log1p(yi) for di, yi in zip(d, y))
    a = torch.full_like(s2, 2.0)
    for _ in range(4):
        g, dg = -a * s2, -s2
        for fi, di, yi in zip(f, d, y):
            z = a * yi
            ph = 1.0 / (13 * 14)
            for k in range(13, 1, -1):
                ph = 1.0 / (k * (k - 1)) - z * ph
            lz = torch.log1p(z)
            g = g + fi * torch.where(z.abs() < 0.05, z * z * ph, (1.0 + z) * lz - z)
            dg = dg + di * lz
        a = torch.where(dg != 0, a - g / dg, a)
    return a


def _stress_tau(f, rho, u, tau, c):
    """Relaxation time of Smagorinsky (1) or eq. (7) (2) from the stress."""
    P = [[sum(e[a] * e[b] * fi for e, fi in zip(C2, f) if e[a] * e[b]) - rho * u[a] * u[b] -
          (rho / 3.0 if a == b else 0.0) for b in range(2)] for a in range(2)]
    tr2 = sum(P[a][b] * P[a][b] for a in range(2) for b in range(2))
    if c["collision"] == 1:
        return 0.5 * (tau + torch.sqrt(tau * tau + 18.0 * c["Cs"] * torch.sqrt(tr2) / rho))
    tr3 = sum(P[a][b] * P[b][e] * P[e][a] for a in range(2) for b in range(2) for e in range(2))
    return torch.where(tr2 == 0, tau + 0 * tr2, tau + tau * tr3 / (2.0 * rho * tr2))


class _Model:
    """The step of eq. (1) on lists of populations [..., (nz,) ny, nx]."""

    def __init__(self, q, tau, alpha, collision=0, case=None, ext=None, damp=0.0):
        self.cs, self.ws = _lattice(q)
        self.tau, self.alpha, self.collision, self.case = tau, alpha, collision, case
        self.ext, self.damp = ext, damp

    def external(self, rho, j):
        ext = list(self.ext)
        if self.damp:  # minus FR0 times the projection of u on the modes 1 <= |k| <= 2
            ny, nx = rho.shape[-2:]
            x = 2.0 * math.pi * torch.arange(nx, dtype=torch.float64, device=rho.device) / nx
            y = 2.0 * math.pi * torch.arange(ny, dtype=torch.float64, device=rho.device)[:, None] / ny
            for a in range(2):
                u = j[a] / rho
                for kx, ky in ((1, 0), (0, 1), (1, 1), (1, -1), (2, 0), (0, 2)):
                    for w in (torch.cos(kx * x + ky * y), torch.sin(kx * x + ky * y)):
                        ext[a] = ext[a] - 2.0 * self.damp * (u * w).mean((-2, -1), keepdim=True) * w
        return ext

    def local(self, f):
        """rho, j, the external force and the viscosity of a state."""
        rho, j = _moments(f, self.cs)
        tau = self.tau
        if self.collision in (1, 2):
            tau = _stress_tau(f, rho, [a / rho for a in j], self.tau, self.case)
        elif self.collision == 3:
            u = [a / rho for a in j]
            d = [_entropic_feq(rho, u, c, w) - fi for fi, c, w in zip(f, self.cs, self.ws)]
            tau = 2.0 * self.tau / _entropy_root(f, d)
        return rho, j, self.external(rho, j), (tau - 0.5) / 3.0

    def step(self, f):
        rho, j = _moments(f, self.cs)
        ext = self.external(rho, j)
        u = [a / rho for a in j]
        v = [a + (e - self.alpha * b) / rho for a, e, b in zip(u, ext, j)]
        feq = _entropic_feq if self.collision == 3 else _feq
        still = self.alpha == 0.0 and not self.damp and all(isinstance(e, float) and e == 0.0 for e in ext)
        eq = [feq(rho, u, c, w) for c, w in zip(self.cs, self.ws)]
        if self.collision == 3:
            om = _entropy_root(f, [e - fi for e, fi in zip(eq, f)]) / (2.0 * self.tau)
        elif self.collision:
            om = 1.0 / _stress_tau(f, rho, u, self.tau, self.case)
        else:
            om = 1.0 / self.tau
        out, dims = [], tuple(range(-1, -1 - len(j), -1))
        for fi, e, c, w in zip(f, eq, self.cs, self.ws):
            g = fi + om * (e - fi)
            if not still:
                g = g + feq(rho, v, c, w) - e
            out.append(torch.roll(g, c, dims) if any(c) else g)
        return out


def _D(a, axis):
    """Eq. (18) along x (0), y (1), z (2)."""
    s = 0.0
    for k, w in ((1, 0.8), (2, -0.2), (3, 4.0 / 105.0), (4, -1.0 / 280.0)):
        s = s + w * (torch.roll(a, -k, -1 - axis) - torch.roll(a, k, -1 - axis))
    return s


def _terms(levels, alpha, dim):
    """The 13 term fields from (rho, j, external force, nu) at n, n-1, n-2."""
    def at(lv):
        rho, j, ext, _ = lv
        F = [e - alpha * a for e, a in zip(ext, j)]
        u = [(a + 0.5 * b) / rho for a, b in zip(j, F)]
        if dim == 2:
            w = [None, None, _D(u[1], 0) - _D(u[0], 1)]
        else:
            w = [_D(u[2], 1) - _D(u[1], 2), _D(u[0], 2) - _D(u[2], 0), _D(u[1], 0) - _D(u[0], 1)]
        return rho, F, u, w, 0.5 * rho * sum(a * a for a in u), 0.5 * sum(a * a for a in w if a is not None)
    A = [at(lv) for lv in levels]
    rho, F, u, w, E, Z = A[0]
    nr, R = levels[0][3] * rho, range(dim)
    lhs = [0.5 * (3.0 * A[0][k] - 4.0 * A[1][k] + A[2][k]) for k in (4, 5)]
    del A
    G = [[_D(u[i], k) for k in R] for i in R]
    S = [[G[i][k] + G[k][i] for k in R] for i in R]
    T = [None] * 13
    T[0], T[6] = lhs
    T[1] = -sum(_D(E * u[k], k) for k in R)
    T[2] = -sum(u[k] * _D(rho - 1.0, k) for k in R) / 3.0
    T[3] = sum(u[k] * F[k] for k in R)
    T[4] = -nr * sum(S[i][k] * G[i][k] for i in R for k in R)
    T[5] = sum(_D(nr * sum(u[i] * S[i][k] for i in R), k) for k in R)
    T[7] = -sum(_D(Z * u[k], k) for k in R)
    T[8] = -Z * sum(G[k][k] for k in R)
    a = [b / rho for b in F]
    H = [sum(_D(nr * S[i][k], k) for k in R) / rho for i in R]
    if dim == 2:
        z = w[2]
        T[9] = z * (_D(a[1], 0) - _D(a[0], 1))
        T[10] = H[0] * _D(z, 1) - H[1] * _D(z, 0)
        T[11] = _D(z * H[1], 0) - _D(z * H[0], 1)
        T[12] = torch.zeros_like(z)
    else:
        nx = lambda i: ((i + 1) % 3, (i + 2) % 3)  # noqa: E731
        T[9] = sum(w[i] * (_D(a[nx(i)[1]], nx(i)[0]) - _D(a[nx(i)[0]], nx(i)[1])) for i in R)
        T[10] = sum(H[i] * (_D(w[nx(i)[1]], nx(i)[0]) - _D(w[nx(i)[0]], nx(i)[1])) for i in R)
        T[11] = sum(_D(H[nx(i)[0]] * w[nx(i)[1]] - H[nx(i)[1]] * w[nx(i)[0]], i) for i in R)
        T[12] = sum(w[i] * w[k] * G[i][k] for i in R for k in R)
    return T, u


def _box_mean(a, L, dim):
    """Means over the L^dim boxes at every periodic origin."""
    m = a.mean(tuple(range(-dim, 0)), keepdim=True)
    a = a - m
    for d in range(-dim, 0):
        cs = torch.cumsum(torch.cat([torch.zeros_like(a.narrow(d, 0, 1)), a, a.narrow(d, 0, L - 1)], d), d)
        n = a.shape[d]
        a = cs.narrow(d, L, n) - cs.narrow(d, 0, n)
    return a / float(L) ** dim + m


def _balance(T, u, Ls, origins, dim):
    """Statistics [B, nL, 15, 2]; with u (mean, std) [B, nL, 2] of the boxes'
    Mach number; in 3D every box [B, rows, 15]."""
    B, stats, rows, mach = T[0].shape[0], [], [], []
    for i, L in enumerate(Ls):
        if L > min(T[0].shape[1:]):
            stats.append(torch.full((B, 15, 2), math.nan, dtype=torch.float64, device=T[0].device))
            mach.append(torch.full((B, 2), math.nan, dtype=torch.float64, device=T[0].device))
            continue
        def boxes(f):
            b = _box_mean(f, L, dim)
            if origins is None:
                return b.reshape(B, -1)
            o = torch.as_tensor(origins[i], device=b.device).long()
            return b[(slice(None),) + tuple(o[:, k] for k in range(dim - 1, -1, -1))]
        v = [boxes(t) for t in T]
        for k0, n in ((6, 6), (0, 5)):
            num = (sum(v[k0 + 1 + k] for k in range(n)) - v[k0]).abs()
            mx = v[k0 + 1].abs()
            for k in range(1, n):
                mx = torch.maximum(mx, v[k0 + 1 + k].abs())
            v.insert(0, torch.where(mx == 0, torch.where(num == 0, 0.0 * num, torch.inf + num), num / mx))
            if k0 == 6:
                dz = v.pop(0)
        v.insert(1, dz)
        st = lambda b: torch.stack([b.mean(1), b.std(1, unbiased=False)], -1)  # noqa: E731
        stats.append(torch.stack([st(b) for b in v], 1))
        if dim == 3:
            rows.append(torch.stack(v, -1))
        if u is not None:
            mach.append(st(torch.sqrt(3.0 * boxes(sum(a * a for a in u)))))
    return (torch.stack(stats, 1), torch.cat(rows, 1) if rows else None,
            torch.stack(mach, 1) if mach else None)


def _column(v):
    return torch.tensor(v, dtype=torch.float64, device=DEV)[:, None, None]


def _external2(c, nx, ny, F0):
    """External force fields of a group (the damping of force kind 2 apart)."""
    x = 2.0 * math.pi * torch.arange(nx, dtype=torch.float64, device=DEV) / nx
    y = 2.0 * math.pi * torch.arange(ny, dtype=torch.float64, device=DEV)[:, None] / ny
    if c["force"] == 0:
        return [0.0, 0.0]
    if c["force"] == 1:
        return [_column(F0) * torch.sin(c["kf"] * y), _column(F0) * torch.sin(c["kf"] * x)]
    fx = fy = 0.0
    for ky in range(0, 8):
        for kx in range(-7, 8):
            if 25 <= kx * kx + ky * ky <= 49 and (ky > 0 or kx > 0):
                s = torch.sin(kx * x + ky * y)
                fx, fy = fx - 2.0 * math.pi * ky / ny * s, fy + 2.0 * math.pi * kx / nx * s
    return [_column(F0) * fx, _column(F0) * fy]


def _advance(model, f, steps):
    """The last state and the levels (rho, j, force, nu) at n, n-1, n-2."""
    levels = []
    for k in range(steps + 1):
        if k >= steps - 2:
            levels.insert(0, model.local(f))
        if k < steps:
            f = model.step(f)
    return f, levels


def _adjoint_f0(c, seed):
    rho, ux, uy = _random_phase(c["nx"], c["ny"], _gen(seed), 0.02)
    return torch.stack([_feq(rho, [ux, uy], e, w) for e, w in zip(C2, W2)])


def _exact_adjoint(c, seed):
    f0 = _adjoint_f0(c, seed).requires_grad_()
    tau = torch.tensor(c["tau"], dtype=torch.float64, device=DEV, requires_grad=True)
    F0 = torch.tensor(_laminar_F0(max(c["nx"], c["ny"]), c["tau"], c["kf"], c["alpha"], c["u"]),
                      dtype=torch.float64, device=DEV, requires_grad=True)
    s = [torch.sin(c["kf"] * 2.0 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n)
         for n in (c["ny"], c["nx"])]
    s[0] = s[0][:, None]
    L, at = c["L"], {}
    for k, n in ((0, c["ny"]), (1, c["nx"])):
        at[k] = torch.arange(-4, c["L"] + 4, device=DEV) % n

    def objective(f, tau, F0):
        r, j = _moments([g[at[0]][:, at[1]] for g in f], C2)
        sx, sy = s[0][at[0]], s[1][at[1]]
        u = [(a + 0.5 * (F0 * e - c["alpha"] * a)) / r for a, e in zip(j, (sx, sy))]
        G = [[_D(a, k)[4:-4, 4:-4] for k in range(2)] for a in u]
        q = sum((G[i][k] + G[k][i]) * G[i][k] for i in range(2) for k in range(2))
        return (-(tau - 0.5) / 3.0 * r[4:-4, 4:-4] * q).mean()

    def part(n, m, tau, F0, *f):
        J = torch.zeros((), dtype=torch.float64, device=DEV)
        for k in range(n, m):
            if k >= c["n0"]:
                J = J + objective(f, tau, F0)
            if k < c["n1"]:
                f = _Model(9, tau, c["alpha"], ext=[F0 * s[0], F0 * s[1]]).step(list(f))
        return (J, *f)

    from torch.utils.checkpoint import checkpoint
    f, J, n, last = list(f0.unbind(0)), 0.0, 0, c["n1"] + 1
    while n < last:
        m = min(n + 25, last)
        got = checkpoint(part, n, m, tau, F0, *f, use_reentrant=False)
        J, f, n = J + got[0], list(got[1:]), m
    J = J / (c["n1"] - c["n0"] + 1)
    J.backward()
    return {"J": J.detach(), "dtau": tau.grad, "dF0": F0.grad, "df0": f0.grad}


def exact(case, seed):
    c = case
    if c["kind"] == "adjoint":
        return _exact_adjoint(c, seed)
    with torch.no_grad():
        if c["kind"] == "d3":
            n = {0: c["nx"], 1: c["ny"], 2: c["nz"]}
            sn = [torch.sin(2.0 * math.pi * c["kf"] * torch.arange(n[a], dtype=torch.float64, device=DEV) / n[a])
                  for a in range(3)]
            F0 = _F0_3(c)
            ext = [F0 * sn[1][:, None], F0 * sn[2][:, None, None], F0 * sn[0]] if c["force"] else [0.0] * 3
            model = _Model(c["lattice"], c["tau"], c["alpha"], ext=ext)
            stats, boxes = [], []
            origins = _origins(c, seed, min(n.values()), 3)
            for rho, *u in _fields3(c, seed):
                f = [_feq(rho, u, e, w) for e, w in zip(model.cs, model.ws)]
                f, levels = _advance(model, f, c["steps"])
                levels = [(r[None], [a[None] for a in j], e, nu) for r, j, e, nu in levels]
                st, rows, _ = _balance(_terms(levels, c["alpha"], 3)[0], None, _ints(c["sizes"]), origins, 3)
                stats.append(st[0].cpu().numpy())
                boxes.append(rows[0])
            return {"stats": np.stack(stats), "boxes": boxes}
        stats, state, mach = [], [], []
        groups, Ls = _groups(c), _ints(c["sizes"])
        origins = _origins(c, seed, min(min(nx, ny) for nx, ny, _, _ in groups))
        for (nx, ny, taus, F0), (rho, ux, uy) in zip(groups, _fields(c, seed)):
            model = _Model(9, _column(taus), c["alpha"], c["collision"], c, _external2(c, nx, ny, F0), c["FR0"])
            f = [_feq(rho, [ux, uy], e, w) for e, w in zip(C2, W2)]
            del rho, ux, uy
            f, levels = _advance(model, f, c["steps"])
            if c["state"] == "populations":
                state.append(torch.stack(f, 1))
            del f
            T, u = _terms(levels, c["alpha"], 2)
            if c["state"] == "moments":
                w = _D(u[1], 0) - _D(u[0], 1)
                state += [{"rho": levels[0][0][b], "ux": u[0][b], "uy": u[1][b], "omega": w[b]}
                          for b in range(len(taus))]
            del levels
            st, _, ma = _balance(T, u if c["hist"] else None, Ls, origins, 2)
            stats.append(st)
            mach.append(ma)
            del T, u
        out = {"stats": torch.cat(stats, 0).cpu().numpy(), "state": state}
        if c["hist"]:  # counts of boxes per bin: whole numbers
            out |= {"mach": torch.cat(mach, 0).cpu().numpy(), "delta_hist": None, "mach_hist": None}
        return out


if __name__ == "__main__":
    for case in listed() + [draw(random.Random(k)) for k in range(6)]:
        print(case, work(case))
