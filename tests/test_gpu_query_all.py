"""Every periodic origin at once (planar tables, chained boxes) against the same
origins given as a list (record tables, four corners per box): the box sums
are exact integers on both paths.  FP32 boxes are then the same bit for bit;
FP64 boxes differ by the one rounding of mean + deviation (bar 1e-15 of the
field's largest box, its propagation through the quotient for the errors).
Sizes at the edges: one column, less and more than a CTA's columns, chains
that close on the edge or wrap, L = 1, L = the grid, L of more than half."""
import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_1809_06735_gb300 as P
    return P


def _lattice(P, nx, ny, prec):
    lat = P.Lattice([P.Member(nx, ny, 0.56, 1.0, 1, 2, 1e-4, 1e-4)], precision=prec, diag_every=4)
    f = [li.smooth_fields(nx, ny, k, amp=a) for k, a in enumerate((.01, .03, .03))]
    lat.init_fields(0, 1.0 + f[0], f[1], f[2])
    lat.step(4)
    return lat


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("nx,ny", [(257, 19), (33, 70), (20, 300), (8, 8), (5, 3), (1, 1), (300, 33),
                                   (129, 64), (520, 40)])
def test_all_origins_equal_the_list(P, nx, ny, prec):
    lat = _lattice(P, nx, ny, prec)
    n = min(nx, ny)
    Ls = sorted({1, 2, 3, n // 2, n // 2 + 1, n - 1, n} & set(range(1, n + 1)))
    y, x = np.mgrid[0:ny, 0:nx]
    org = np.stack([x.ravel(), y.ravel()], 1).astype(np.int32)
    sa, ba = lat.subvolume_balance(0, Ls, per_box=True)
    sl, bl = lat.subvolume_balance(0, Ls, origins=org, per_box=True)
    ba, bl = ba.cpu().numpy(), bl.cpu().numpy()
    assert ba.shape == bl.shape
    if prec == 32:
        assert np.array_equal(ba, bl, equal_nan=True)
        np.testing.assert_allclose(sa[:, 2:], sl[:, 2:], rtol=2e-5, atol=1e-5 * np.max(np.abs(sl[:, 2:])))
    else:
        scale = np.max(np.abs(bl[:, 2:]), axis=0)
        assert np.all(np.abs(ba[:, 2:] - bl[:, 2:]) <= 1e-15 * scale + 4e-16 * np.abs(bl[:, 2:]))
        for q, k in ((0, 2), (1, 8)):  # 7 roundings of the terms over the largest right-hand side
            mx = np.max(np.abs(bl[:, k + 1:k + 6]), axis=1)
            with np.errstate(divide="ignore", invalid="ignore"):
                bar = 20 * 1e-15 * np.sum(scale[k - 2:k + 4]) / mx + 1e-15 * np.abs(bl[:, q])
            ok = (ba[:, q] == bl[:, q]) | (np.abs(ba[:, q] - bl[:, q]) <= bar) | (mx == 0)
            assert np.all(ok)
    lat.close()


def test_distributions_equal_the_list(P):
    """Histograms over every origin: the counts of the same origins as a list."""
    lat = _lattice(P, 131, 77, 32)
    y, x = np.mgrid[0:77, 0:131]
    org = np.stack([x.ravel(), y.ravel()], 1).astype(np.int32)
    de, me = np.linspace(0, 0.5, 33), np.linspace(0, 0.2, 17)
    a = lat.subvolume_distributions([0], [1, 4, 40, 77], de, me)
    b = lat.subvolume_distributions([0], [1, 4, 40, 77], de, me, origins=org)
    assert np.array_equal(a["delta_hist"], b["delta_hist"])
    assert np.array_equal(a["mach_hist"], b["mach_hist"])
    assert np.all(a["mach_hist"].sum(-1) == 131 * 77)
    np.testing.assert_allclose(a["mach"], b["mach"], rtol=1e-5, atol=1e-9)
    lat.close()


@pytest.mark.parametrize("nx,ny", [(1000, 1000), (512, 512), (260, 260)])
def test_sizes_together_equal_sizes_alone(P, nx, ny):
    """Sizes of nearly the whole grid use another number of CTAs than the
    rest: the partial sums of one size must not reach another's.  FP32: the
    CTAs of a size do not depend on the other sizes, so the same bits."""
    lat = _lattice(P, nx, ny, 32)
    Ls = [2, 10, nx // 3, nx - 1, nx]
    s = lat.subvolume_balance(0, Ls)
    for i, L in enumerate(Ls):
        assert np.array_equal(s[i], lat.subvolume_balance(0, [L])[0], equal_nan=True), L
