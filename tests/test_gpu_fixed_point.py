"""The FP64 step's fixed-point collision against the FP64 oracle at the edges
of its range, where it hands cells over to the FP64 form: densities over the
whole octave of its scale, tiny and negative populations, fast cells, strong
forces, relaxation times near 1/2 and far above, and non-finite values.
Bar: 1e-12 relative on the populations, as for every FP64 step."""
import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_1809_06735_gb300 as P
    return P


def _run(P, f0, steps, tau, rho0, force, storage=2):
    ny, nx = f0.shape[1:]
    kind, F0, kf, alpha = force
    lat = P.Lattice([P.Member(nx, ny, tau, rho0, kind, kf, F0, alpha)], precision=64, storage=storage)
    lat.set_populations(0, f0)
    lat.step(steps)
    out = lat.get_populations_host(0)
    lat.close()
    return out


@pytest.mark.parametrize("rho0", [1.0, 1.999, 0.75, 3e-5, 4.1e6])
@pytest.mark.parametrize("tau", [0.5001, 0.56, 30.0])
@pytest.mark.parametrize("forced", [False, True])
def test_densities(P, orc, rho0, tau, forced):
    f0 = rho0 * li.random_populations(37, 23, seed=3, rel_noise=0.02)
    force = (1, 3e-4 * rho0, 2, 1e-3) if forced else (0, 0.0, 0, 0.0)
    got = _run(P, f0, 10, tau, rho0, force)
    ref = orc.run(f0, 10, tau, orc.Force(force[0], force[1], force[2], force[3]))
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-12


@pytest.mark.parametrize("storage", [1, 2])
def test_cells_outside_the_range(P, orc, storage):
    """Cells that take the FP64 form beside cells that do not: after one step
    every population is the oracle's to 1e-12 of its cell's density."""
    f0 = li.random_populations(40, 30, seed=4, rel_noise=0.02)
    f0[5, 3, :] = 1e-7          # below the range
    f0[2, 7, ::3] = 0.0
    f0[6, 9, 5] = -1e-3         # negative
    f0[1, 12, :] *= 6.0         # fast: |u| about 0.4
    f0[0, 15, 4] = 3.0          # dense
    f0[3, 20, 7] = 1e-300
    got = _run(P, f0, 1, 0.7, 1.0, (1, 0.3, 2, 1e-3), storage)  # |F| / rho above 1/8 too
    ref = orc.run(f0, 1, 0.7, orc.Force(1, 0.3, 2, 1e-3))
    assert np.max(np.abs(got - ref)) < 1e-12 * np.max(f0.sum(0))


def test_non_finite_cells_spread_as_before(P):
    """A NaN and an infinity reach their neighbours and are flagged."""
    f0 = li.random_populations(32, 32, seed=5, rel_noise=0.01)
    f0[4, 8, 8] = np.nan
    f0[1, 20, 20] = np.inf
    lat = P.Lattice([P.Member(32, 32, 0.6)], precision=64)
    lat.set_populations(0, f0)
    lat.step(1)
    g = lat.get_populations_host(0)
    assert lat.member_status(0) == 1
    bad = ~np.isfinite(g).all(0)
    want = np.zeros((32, 32), bool)
    want[7:10, 7:10] = want[19:22, 19:22] = True
    assert np.array_equal(bad, want)
    lat.close()


@pytest.mark.parametrize("rho0", [1.0, 1.999, 0.75, 3e-5, 4.1e6])
@pytest.mark.parametrize("grids", [[(255, 128)], [(256, 128)], [(331, 103)], [(40, 30), (256, 128)]])
def test_both_sides_of_the_size_rule(P, orc, rho0, grids):
    """Grids below 2^15 cells take the FP64 form, those from it up the fixed
    point, also side by side in one launch; a few cells are outside its range.
    1e-12 of the cells' density, as above."""
    mem = [P.Member(nx, ny, 0.56, rho0, 1, 2, 3e-4 * rho0, 1e-3) for nx, ny in grids]
    lat = P.Lattice(mem, precision=64)
    f0 = []
    for m, (nx, ny) in enumerate(grids):
        f = rho0 * li.random_populations(nx, ny, seed=m, rel_noise=0.02)
        f[5, 3, :4] = 1e-7 * rho0
        f[0, 15, 4] = 3.0 * rho0
        f0.append(f)
        lat.set_populations(m, f)
    lat.step(5)
    for m, f in enumerate(f0):
        ref = orc.run(f, 5, 0.56, orc.Force(1, 3e-4 * rho0, 2, 1e-3))
        assert np.max(np.abs(lat.get_populations_host(m) - ref)) < 1e-12 * np.max(f.sum(0))
    lat.close()
