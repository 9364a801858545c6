"""Whole gradients of the box-averaged dissipation against extended precision: the
model and the objective in numpy's long double with the complex-step method (no
differences), on a grid that steps in fixed point and one that does not.
tests/golden/gradients_extended.json holds J, dJ/dtau, dJ/dF0 and dJ/df0 . d for
a fixed direction d; running this file writes it anew where long double has 64
bits of significand.

Bars: 200 steps of one rounding each (2^-53), four times over for the quadratic
objective, once for J and once more for the adjoint's own roundings: 1e-13 and
2e-13 of the value (of the sum of the products' magnitudes for dJ/df0 . d); the force is held to 2^-62 of the density in the fixed-point step
and the adjoint (1.4e-14 of F0 = 1.5e-5), well inside."""
import json
import os

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
GOLDEN = os.path.join(HERE, "golden", "gradients_extended.json")
GRIDS = {"256x130": (256, 130), "48x40": (48, 40)}
TAU, F0, ALPHA, KF, L, N0, N1 = 0.55, 1.5e-5, 1e-4, 2, 12, 100, 200
CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)


def _inputs(nx, ny, orc):
    """Populations of a smooth flow and a direction, the same bits on every machine."""
    def wave(n, k, ph):
        return np.round(np.sin(2.0 * np.pi * (k * np.arange(n) / n + ph)) * 2.0 ** 40) / 2.0 ** 40

    ux = 0.03 * (wave(nx, 2, 0.1)[None, :] * wave(ny, 3, 0.6)[:, None] + 0.5 * wave(ny, 1, 0.3)[:, None])
    uy = 0.03 * (wave(nx, 1, 0.8)[None, :] * wave(ny, 2, 0.2)[:, None] + 0.5 * wave(nx, 3, 0.4)[None, :])
    rho = 1.0 + 0.002 * wave(nx, 1, 0.45)[None, :] * wave(ny, 1, 0.05)[:, None]
    d = np.stack([wave(nx, l + 1, 0.07 * l)[None, :] * wave(ny, 9 - l, 0.11 * l)[:, None] for l in range(9)])
    return orc.init(rho, ux, uy), d


@pytest.mark.gpu
@pytest.mark.parametrize("grid", sorted(GRIDS))
def test_gradients(orc, grid):
    import torch

    from paper_1809_06735_gb300 import adjoint
    with open(GOLDEN) as fh:
        want = json.load(fh)[grid]
    nx, ny = GRIDS[grid]
    f, d = _inputs(nx, ny, orc)
    spec = adjoint.ObjectiveSpec(nx, ny, KF, ALPHA, N0, N1, (nx - 5, 3), L, 64, 50)
    f0 = torch.from_numpy(f).cuda().requires_grad_()
    tau = torch.tensor(TAU, dtype=torch.float64, requires_grad=True)
    amp = torch.tensor(F0, dtype=torch.float64, requires_grad=True)
    J = adjoint.box_dissipation(tau, amp, f0, spec)
    J.backward()
    gd = f0.grad.cpu().numpy().astype(np.longdouble) * d
    got = {"J": float(J.detach()), "dtau": float(tau.grad), "dF0": float(amp.grad), "df0.d": float(np.sum(gd))}
    for k, v in got.items():
        size = float(np.sum(np.abs(gd))) if k == "df0.d" else abs(want[k])
        print("%s %s: off by %.1e" % (grid, k, abs(v - want[k]) / size))
        assert abs(v - want[k]) <= (1e-13 if k == "J" else 2e-13) * size, (k, v, want[k])


def _objective(f, tau, amp, nx, ny):
    """J in the arithmetic of f, tau and amp (long double, complex or not)."""
    LD = np.longdouble
    om, al = 1 / tau, LD(ALPHA)
    T = [LD(4) / 9] + [LD(1) / 9] * 4 + [LD(1) / 36] * 4
    sx = np.sin(2 * np.pi * KF * np.arange(ny) / ny).astype(LD)[:, None]
    sy = np.sin(2 * np.pi * KF * np.arange(nx) / nx).astype(LD)[None, :]
    box = np.ix_(np.arange(3 - 4, 3 + L + 4) % ny, np.arange(nx - 5 - 4, nx - 5 + L + 4) % nx)
    co = [LD(8) / 10, -LD(2) / 10, LD(4) / 105, -LD(1) / 280]

    def D(a, k):
        return sum(c * (np.roll(a, -m, 1 - k) - np.roll(a, m, 1 - k)) for m, c in zip((1, 2, 3, 4), co))

    J = 0
    for n in range(N1 + 1):
        r = f.sum(0)
        jx, jy = (sum(c[l] * f[l] for l in range(9) if c[l]) for c in (CX, CY))
        if n >= N0:
            u = [((jx + LD(.5) * (amp * sx - al * jx)) / r)[box], ((jy + LD(.5) * (amp * sy - al * jy)) / r)[box]]
            G = [[D(a, k) for k in range(2)] for a in u]
            q = sum((G[i][k] + G[k][i]) * G[i][k] for i in range(2) for k in range(2))
            J = J + ((-(tau - LD(.5)) / 3 * r[box] * q)[4:-4, 4:-4]).mean()
        if n == N1:
            return J / (N1 - N0 + 1)
        mx, my, ir = (1 - al) * jx + amp * sx, (1 - al) * jy + amp * sy, 1 / r
        a2, b2 = LD(1.5) * (jx * jx + jy * jy) * ir, LD(1.5) * (mx * mx + my * my) * ir
        g = np.empty_like(f)
        for l in range(9):
            ca, cb = CX[l] * jx + CY[l] * jy, CX[l] * mx + CY[l] * my
            fa = T[l] * (r + 3 * ca + LD(4.5) * ca * ca * ir - a2)
            fb = T[l] * (r + 3 * cb + LD(4.5) * cb * cb * ir - b2)
            g[l] = np.roll((1 - om) * f[l] + (om - 1) * fa + fb, (CY[l], CX[l]), (0, 1))
        f = g


def _write_golden():
    import sys
    sys.path.insert(0, os.path.dirname(HERE))
    import oracle as orc
    C, h = np.clongdouble, np.longdouble(1e-40)
    assert np.finfo(np.longdouble).nmant == 63, "the reference needs x87 long doubles"
    out = {}
    for name, (nx, ny) in GRIDS.items():
        f, d = _inputs(nx, ny, orc)
        f, t, a = f.astype(C), C(TAU), C(F0)
        J = _objective(f, t + 1j * h, a, nx, ny)
        out[name] = {"J": float(J.real), "dtau": float(J.imag / h),
                     "dF0": float(_objective(f, t, a + 1j * h, nx, ny).imag / h),
                     "df0.d": float(_objective(f + 1j * h * d, t, a, nx, ny).imag / h)}
    with open(GOLDEN, "w") as fh:
        json.dump(out, fh, indent=1)


if __name__ == "__main__":
    _write_golden()
