"""The FP64 step's fixed-point collision on grids that take it (2^15 cells and
more, here 331 x 103 and 182 x 181, which no block divides): one step against
exact rational arithmetic, which tells it from the FP64 form, and the edges of
its range, where it hands cells over to the FP64 form, against the oracle:
densities over the octave of its scale, relaxation times near 1/2 and far above,
tiny, zero, negative and fast cells, strong forces, non-finite values, in both
storages (the in-place one reads the cell again for the FP64 form).

Bars.  One step: the final rounding (2^-53 of the population) and about four units
of 2^-64 in a population of at least 2^-7.9 (5e-17): 2^-52 relative; the FP64
form is off by up to 1.2e-15.  Several steps and cells outside the range: 1e-12, as
for every FP64 step."""
import math
from fractions import Fraction

import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu

NX, NY = 331, 103
C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W = [Fraction(4, 9)] + [Fraction(1, 9)] * 4 + [Fraction(1, 36)] * 4


@pytest.fixture(scope="module")
def P():
    import paper_1809_06735_gb300 as P
    return P


def _run(P, f0, steps, tau, rho0, force, storage):
    ny, nx = f0.shape[1:]
    kind, F0, kf, alpha = force
    lat = P.Lattice([P.Member(nx, ny, tau, rho0, kind, kf, F0, alpha)], precision=64, storage=storage)
    lat.set_populations(0, f0)
    lat.step(steps)
    out, status = lat.get_populations_host(0), lat.member_status(0)
    lat.close()
    return out, status


def _exact_cell(f, omega, alpha, Fx, Fy):
    """The collision of eq. (1) with the exact-difference term, in rationals."""
    rho = sum(f)
    j = [sum(c[a] * v for c, v in zip(C, f)) for a in (0, 1)]
    F = [Fx - alpha * j[0], Fy - alpha * j[1]]

    def feq(u):
        uu = u[0] * u[0] + u[1] * u[1]
        out = []
        for c, w in zip(C, W):
            cu = c[0] * u[0] + c[1] * u[1]
            out.append(w * rho * (1 + 3 * cu + Fraction(9, 2) * cu * cu - Fraction(3, 2) * uu))
        return out

    e0 = feq([a / rho for a in j])
    e1 = feq([(a + b) / rho for a, b in zip(j, F)])
    return [v - omega * (v - a) + b - a for v, a, b in zip(f, e0, e1)]


@pytest.mark.parametrize("storage", [1, 2])
@pytest.mark.parametrize("rho0", [1.0, 1.999, 0.75, 3e-5, 4.1e6])
@pytest.mark.parametrize("tau", [0.5001, 0.56, 30.0])
@pytest.mark.parametrize("forced", [False, True])
def test_one_step_is_exact_to_the_rounding(P, rho0, tau, forced, storage):
    f0 = rho0 * li.random_populations(NX, NY, seed=3, rel_noise=0.02)
    kind, F0, kf, alpha = (1, 3e-4 * rho0, 2, 1e-3) if forced else (0, 0.0, 0, 0.0)
    got, _ = _run(P, f0, 1, tau, rho0, (kind, F0, kf, alpha), storage)
    rng = np.random.default_rng(7)
    worst = 0.0
    for y, x in zip(rng.integers(0, NY, 100), rng.integers(0, NX, 100)):
        Fx = F0 * math.sin(2.0 * math.pi * kf * float(y) / NY) if forced else 0.0
        Fy = F0 * math.sin(2.0 * math.pi * kf * float(x) / NX) if forced else 0.0
        ref = _exact_cell([Fraction(float(v)) for v in f0[:, y, x]], Fraction(1.0 / tau),
                          Fraction(alpha), Fraction(Fx), Fraction(Fy))
        for l, (cx, cy) in enumerate(C):
            v = Fraction(float(got[l, (y + cy) % NY, (x + cx) % NX]))
            worst = max(worst, float(abs(v - ref[l]) / ref[l]))
    assert worst < 2.0 ** -52


@pytest.mark.parametrize("storage", [1, 2])
@pytest.mark.parametrize("rho0", [1.0, 1.999, 0.75, 3e-5, 4.1e6])
@pytest.mark.parametrize("tau", [0.5001, 0.56, 30.0])
@pytest.mark.parametrize("forced", [False, True])
def test_densities(P, orc, rho0, tau, forced, storage):
    f0 = rho0 * li.random_populations(NX, NY, seed=3, rel_noise=0.02)
    force = (1, 3e-4 * rho0, 2, 1e-3) if forced else (0, 0.0, 0, 0.0)
    got, _ = _run(P, f0, 9, tau, rho0, force, storage)
    ref = orc.run(f0, 9, tau, orc.Force(force[0], force[1], force[2], force[3]))
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-12


@pytest.mark.parametrize("storage", [1, 2])
@pytest.mark.parametrize("nx,ny", [(NX, NY), (182, 181)])
@pytest.mark.parametrize("F0", [0.0, 3e-4, 0.3])
def test_cells_outside_the_range(P, orc, nx, ny, F0, storage):
    """One step in each phase of the storage; F0 = 0.3 takes |F| / rho above 1/8."""
    f0 = li.random_populations(nx, ny, seed=4, rel_noise=0.02)
    f0[5, 3, :] = 1e-7          # below the range
    f0[2, 7, ::3] = 0.0
    f0[6, 9, 5] = -1e-3         # negative
    f0[1, 12, :] *= 6.0         # fast: |u| about 0.4
    f0[0, 15, 4] = 3.0          # dense
    f0[3, 20, 7] = 1e-300
    force = (1, F0, 2, 1e-3) if F0 else (0, 0.0, 0, 0.0)
    for steps in (1, 2):
        got, _ = _run(P, f0, steps, 0.7, 1.0, force, storage)
        ref = orc.run(f0, steps, 0.7, orc.Force(force[0], force[1], force[2], force[3]))
        assert np.max(np.abs(got - ref)) < 1e-12 * np.max(f0.sum(0)), steps


@pytest.mark.parametrize("storage", [1, 2])
def test_non_finite_cells_spread_as_before(P, storage):
    f0 = li.random_populations(NX, NY, seed=5, rel_noise=0.01)
    f0[4, 8, 8] = np.nan
    f0[1, 20, 20] = np.inf
    f0[2, 60, 300] = -np.inf
    got, status = _run(P, f0, 1, 0.6, 1.0, (0, 0.0, 0, 0.0), storage)
    assert status == 1
    want = np.zeros((NY, NX), bool)
    want[7:10, 7:10] = want[19:22, 19:22] = want[59:62, 299:302] = True
    assert np.array_equal(~np.isfinite(got).all(0), want)
