"""Several time steps per launch (temporal blocking) against the single-step
kernel, bit for bit: the arithmetic of a cell and its order are the same, only
where the intermediate populations are kept differs.  Sizes at the edges of
the kernel's tiles: one active lane, one warp less and more than a whole row,
whole rows of 1 to 8 warps, strips with halos, blocks that do not divide ny,
ny smaller than a block's recomputed rows."""
import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu

GRIDS = [(512, 64), (132, 70), (1028, 30), (4, 9), (640, 50), (64, 4), (892, 33), (384, 51),
         (256, 65), (1024, 40), (8, 8), (128, 5), (124, 64), (300, 40)]


@pytest.fixture(scope="module")
def P():
    import paper_1809_06735_gb300 as P
    return P


def rel_err(got, want):
    return np.max(np.abs(got - want) / np.abs(want))


def _pair(P, members, T, rows, **kw):
    """The same members with T steps per launch and with single steps."""
    out = []
    for steps in (T, 1):
        lat = P.Lattice(members, precision=32, storage=2, **kw)
        lat.set_steps_per_launch(steps, rows)
        assert lat.steps_per_launch == steps
        for m, mb in enumerate(members):
            f = [li.smooth_fields(mb.nx, mb.ny, 3 * m + k, amp=a) for k, a in enumerate((.01, .03, .03))]
            lat.init_fields(m, 1.0 + f[0], f[1], f[2])
        out.append(lat)
    return out


@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("T,rows", [(2, 8), (3, 8), (4, 8), (2, 100), (3, 27), (4, 100)])
def test_equals_single_steps(P, T, rows, forced):
    kw = dict(force_kind=1, kf=2, F0=1e-5, alpha=1e-4) if forced else {}
    members = [P.Member(nx, ny, 0.53 + 0.01 * i, **kw) for i, (nx, ny) in enumerate(GRIDS)]
    a, b = _pair(P, members, T, rows)
    for n in (1, 2, 3, 4, 5, 7, 12):
        a.step(n)
        b.step(n)
        for m in range(len(members)):
            assert np.array_equal(a.get_populations_host(m), b.get_populations_host(m)), (n, GRIDS[m])
    a.close()
    b.close()


@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("T,rows", [(2, 8), (3, 27), (4, 100)])
def test_entropic_equals_single_steps(P, T, rows, forced):
    """The entropic collision likewise, with members whose cells are close to
    equilibrium, far from it (the root iterated) and at rest."""
    kw = dict(force_kind=1, kf=2, F0=1e-5, alpha=1e-4) if forced else {}
    members = [P.Member(nx, ny, 0.52, collision=3, **kw) for nx, ny in ((132, 70), (256, 65), (8, 8))]
    a, b = _pair(P, members, T, rows)
    far = li.random_populations(256, 65, seed=4, rel_noise=0.04)
    rest = np.tile(li.random_populations(1, 1, seed=1, rel_noise=0.0), (1, 8, 8))
    for lat in (a, b):
        lat.set_populations(1, far)
        lat.set_populations(2, rest)
    for n in (1, 2, 3, 5):
        a.step(n)
        b.step(n)
        for m in range(3):
            assert np.array_equal(a.get_populations_host(m), b.get_populations_host(m)), (n, m)
    a.close()
    b.close()


@pytest.mark.parametrize("graph", [0, 5, 6])
def test_snapshots_and_graphs(P, graph):
    """Snapshot steps, graph replay and remainders around them."""
    members = [P.Member(256, 65, 0.55, 1.0, 1, 2, 1e-5, 1e-4), P.Member(132, 70, 0.6)]
    a, b = _pair(P, members, 3, 16, diag_every=20, graph_steps=graph)
    for n in (20, 33, 7):
        a.step(n)
        b.step(n)
        assert a.time == b.time
        for m in range(2):
            assert np.array_equal(a.get_populations_host(m), b.get_populations_host(m))
    assert a.time == 60
    assert np.array_equal(a.subvolume_balance_batch([0, 1], [2, 16]),
                          b.subvolume_balance_batch([0, 1], [2, 16]))
    assert a.launch_count < b.launch_count
    a.close()
    b.close()


def test_against_the_oracle(P):
    """100 steps within the FP32 population bar (2e-6 relative)."""
    import oracle as orc
    m = P.Member(132, 70, 0.56, 1.0, 1, 2, 1e-5, 1e-4)
    lat = P.Lattice([m], precision=32, storage=2)
    lat.set_steps_per_launch(3, 24)
    f0 = li.random_populations(132, 70, seed=9, rel_noise=0.01)
    lat.set_populations(0, f0)
    lat.step(100)
    ref = orc.run(f0, 100, 0.56, orc.Force(1, 1e-5, 2, 1e-4))
    assert rel_err(lat.get_populations_host(0), ref) < 2e-6


def test_refusals(P):
    """What several steps per launch cannot take is refused and the setting kept."""
    for members, kw in (([P.Member(64, 64, 0.6)], dict(storage=1)),
                        ([P.Member(66, 64, 0.6)], dict(storage=2)),
                        ([P.Member(64, 3, 0.6)], dict(storage=2)),
                        ([P.Member(64, 64, 0.6, collision=1, Cs=0.1)], dict(storage=2)),
                        ([P.Member(64, 64, 0.6, 1.0, 2, 0, 1e-5)], dict(storage=2))):
        lat = P.Lattice(members, precision=32, **kw)
        with pytest.raises(P.LBMError):
            lat.set_steps_per_launch(2)
        lat.set_steps_per_launch(1)
        assert lat.steps_per_launch == 1
        lat.close()
    lat = P.Lattice([P.Member(64, 64, 0.6)], precision=32, storage=2)
    for steps, rows in ((0, 64), (5, 64), (2, 7)):
        with pytest.raises(P.LBMError):
            lat.set_steps_per_launch(steps, rows)
    lat.set_steps_per_launch(4, 8)
    assert lat.steps_per_launch == 4
    lat.set_launch(8, 1)
    assert lat.steps_per_launch == 1
    lat.close()


@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("T,rows", [(2, 8), (3, 27), (4, 100)])
def test_entropic_far_cells_at_the_rim(P, T, rows, forced):
    """Cells whose root is iterated in rows that no warp width divides and in
    strips with halos: lanes past the row and the rims of the strips iterate
    nothing, every stored cell does."""
    kw = dict(force_kind=1, kf=2, F0=1e-5, alpha=1e-4) if forced else {}
    grids = ((132, 70), (392, 33), (1500, 20), (4, 40))
    members = [P.Member(nx, ny, 0.52, collision=3, **kw) for nx, ny in grids]
    a, b = _pair(P, members, T, rows)
    for lat in (a, b):
        for m, (nx, ny) in enumerate(grids):
            lat.set_populations(m, li.random_populations(nx, ny, seed=m, rel_noise=0.04))
    for n in (1, 2, 3, 5):
        a.step(n)
        b.step(n)
        for m in range(len(grids)):
            assert np.array_equal(a.get_populations_host(m), b.get_populations_host(m)), (n, m)
    a.close()
    b.close()
