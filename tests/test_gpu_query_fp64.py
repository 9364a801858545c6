"""The FP64 query over every periodic origin of grids from 2^15 cells up (planar
tables, integer sums of deviations), which smaller FP64 grids do not take:
every box against the same origins given as a list (record tables), the means
and standard deviations against those of the boxes, the distributions against
the list's counts, and batches in which members with planar tables and members
with record tables meet.

Bars, from the arithmetic: a term's box is the same integer on both paths, so it
differs by the rounding of mean + deviation (1e-15 of the largest box); its
standard deviation is summed from integers, so it differs from numpy's by the
rounding of the boxes (1e-15 of the largest) and of some hundred additions
(1e-12 of itself); the errors' variance is a difference of two sums of squares
(1e-13 of the mean square)."""
import math

import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu

GRIDS = [(257, 131), (131, 257), (400, 90), (1025, 33), (33, 1025), (182, 181), (184, 180)]


@pytest.fixture(scope="module")
def P():
    import paper_1809_06735_gb300 as P
    return P


def _lattice(P, grids, prec=64, terms=0):
    members = [P.Member(nx, ny, 0.56 + 0.02 * i, 1.0, 1, 2, 1e-4, 1e-4) for i, (nx, ny) in enumerate(grids)]
    lat = P.Lattice(members, precision=prec, diag_every=4, diag_precision=terms)
    for m, (nx, ny) in enumerate(grids):
        f = [li.smooth_fields(nx, ny, 5 * m + k, amp=a) for k, a in enumerate((.01, .03, .03))]
        lat.init_fields(m, 1.0 + f[0], f[1], f[2])
    lat.step(4)
    return lat


def _every(nx, ny):
    y, x = np.mgrid[0:ny, 0:nx]
    return np.stack([x.ravel(), y.ravel()], 1).astype(np.int32)


def _sizes(nx, ny):
    n = min(nx, ny)
    return sorted({1, 2, n // 3, n // 2 + 1, n - 1, n})


def _moments(b):
    """Means and standard deviations of the columns of b, summed exactly (numpy adds
    the rows of a C-ordered array one by one: some 1e-13 over 2^15 rows)."""
    mean = np.array([math.fsum(c) / b.shape[0] for c in b.T])
    return mean, np.sqrt([math.fsum(c) / b.shape[0] for c in ((b - mean) ** 2).T])


def _check_stats(stats, boxes, nL):
    boxes = boxes.reshape(nL, -1, 15)
    scale = np.max(np.abs(boxes[:, :, 2:]), axis=(0, 1))
    for i in range(nL):
        b = boxes[i]
        mean, std = _moments(b[:, 2:])
        assert np.all(np.abs(stats[i, 2:, 0] - mean) <= 4e-15 * scale), i
        assert np.all(np.abs(stats[i, 2:, 1] - std) <= 1e-12 * std + 1e-15 * scale), i
        if np.all(np.isfinite(b[:, :2])):
            mean, std = _moments(b[:, :2])
            ms = mean ** 2 + std ** 2
            assert np.all(np.abs(stats[i, :2, 0] - mean) <= 1e-13 * np.sqrt(ms)), i
            assert np.all(np.abs(stats[i, :2, 1] ** 2 - std ** 2) <= 1e-13 * ms), i


@pytest.mark.parametrize("prec,terms", [(64, 0), (32, 64)])
@pytest.mark.parametrize("nx,ny", GRIDS)
def test_boxes_and_statistics(P, nx, ny, prec, terms):
    lat = _lattice(P, [(nx, ny)], prec, terms)
    Ls = _sizes(nx, ny)
    sa, ba = lat.subvolume_balance(0, Ls, per_box=True)
    _, bl = lat.subvolume_balance(0, Ls, origins=_every(nx, ny), per_box=True)
    ba, bl = ba.cpu().numpy(), bl.cpu().numpy()
    scale = np.max(np.abs(bl[:, 2:]), axis=0)
    assert np.all(np.abs(ba[:, 2:] - bl[:, 2:]) <= 1e-15 * scale + 4e-16 * np.abs(bl[:, 2:]))
    _check_stats(sa, ba, len(Ls))
    s = lat.subvolume_balance(0, Ls)  # without the boxes' output
    assert np.array_equal(s, sa, equal_nan=True)
    lat.close()


@pytest.mark.parametrize("nx,ny", [(257, 131), (400, 90), (33, 1025)])
def test_distributions(P, nx, ny):
    lat = _lattice(P, [(nx, ny)])
    Ls = _sizes(nx, ny)
    de, me = np.linspace(0, 0.5, 33), np.linspace(0, 0.2, 17)
    a = lat.subvolume_distributions([0], Ls, de, me)
    b = lat.subvolume_distributions([0], Ls, de, me, origins=_every(nx, ny))
    assert np.array_equal(a["delta_hist"], b["delta_hist"])
    assert np.array_equal(a["mach_hist"], b["mach_hist"])
    assert np.all(a["mach_hist"].sum(-1) == nx * ny)
    np.testing.assert_allclose(a["mach"][..., 0], b["mach"][..., 0], rtol=1e-13)
    _, boxes = lat.subvolume_balance(0, Ls, per_box=True)
    _check_stats(a["stats"][0], boxes.cpu().numpy(), len(Ls))
    lat.close()


@pytest.mark.parametrize("dist", [False, True])
def test_mixed_batches(P, dist):
    """Small grids (records, every size by one kernel), larger ones (planar) and
    one whose only sizes are nearly the whole grid, in one call and alone."""
    grids = [(64, 48), (257, 131), (184, 180), (100, 37), (300, 160)]
    lat = _lattice(P, grids)
    de, me = np.linspace(0, 0.5, 33), np.linspace(0, 0.2, 17)
    for Ls in ([3, 16, 33, 131], [180], [37, 180]):
        if dist:
            got = lat.subvolume_distributions(list(range(5)), Ls, de, me)
            st = got["stats"]
        else:
            st = lat.subvolume_balance_batch(list(range(5)), Ls)
        for m, (nx, ny) in enumerate(grids):
            fit = [i for i, L in enumerate(Ls) if L <= min(nx, ny)]
            for i in set(range(len(Ls))) - set(fit):
                assert np.all(np.isnan(st[m, i]))
            if not fit:
                continue
            own = [Ls[i] for i in fit]
            _, boxes = lat.subvolume_balance(m, own, per_box=True)
            _check_stats(st[m, fit], boxes.cpu().numpy(), len(fit))
            if dist:
                one = lat.subvolume_distributions([m], own, de, me)
                assert np.array_equal(got["delta_hist"][m, fit], one["delta_hist"][0])
                assert np.array_equal(got["mach_hist"][m, fit], one["mach_hist"][0])
    lat.close()
