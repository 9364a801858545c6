"""The FP64 query over every periodic origin in batches in which members with
planar tables (from 2^15 cells up) and members with record tables meet: the means
and standard deviations against those of the boxes, the distributions against
each member's own.

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
