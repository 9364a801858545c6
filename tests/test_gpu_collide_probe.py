"""The exactness that the packed collisions rest on: the Newton-corrected
reciprocal and square root against CUDA's correctly rounded ones, float by float,
and the packed BGK and entropic collisions against the scalar ones, bit for bit,
on cells near equilibrium, at the threshold of the root's series and far from
equilibrium, at rest, with one cell of a pair beyond the series, and non-finite."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
C = np.array([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)])


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1809_06735_gb300 import build
    so = str(tmp_path_factory.mktemp("probe") / "collide_probe.so")
    subprocess.run([build.nvcc(), *build._flags(["-I", build.CSRC, "-shared"]),
                    os.path.join(HERE, "collide_probe.cu"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.probe_count.restype = ctypes.c_longlong
    lib.probe_count.argtypes = [ctypes.c_int, ctypes.c_uint, ctypes.c_uint]
    lib.probe_pairs.argtypes = ([ctypes.c_int] * 2 + [ctypes.c_void_p, ctypes.c_int] +
                                [ctypes.c_float] * 5 + [ctypes.c_void_p] * 3)
    return lib


def _bits(x):
    return int(np.float32(x).view(np.uint32))


@pytest.mark.parametrize("what,lo,hi", [(0, 2.0 ** -100, 2.0 ** 100), (1, 1.0, 4.0)])
def test_newton_is_correctly_rounded(probe, what, lo, hi):
    assert probe.probe_count(what, _bits(lo), _bits(hi)) == 0


def _cells(rho0, amp, noise, n, seed):
    """Deviations from rho0 t of 2 n cells: the equilibrium of velocities up to amp
    plus relative noise, in FP32."""
    rng = np.random.default_rng(seed)
    u = amp * rng.uniform(-1, 1, (2 * n, 2))
    rho = rho0 * (1 + 0.3 * amp * rng.uniform(-1, 1, (2 * n, 1)))
    cu = u @ C.T
    f = rho * W * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * np.sum(u * u, 1, keepdims=True))
    f *= 1 + noise * rng.uniform(-1, 1, f.shape)
    return (f - rho0 * W).astype(np.float32)


def _pairs(probe, elbm, forced, cells, rho0, tau=0.51):
    import torch
    n = cells.shape[0] // 2
    d = torch.from_numpy(np.ascontiguousarray(cells)).cuda()
    a, b = torch.empty_like(d), torch.empty_like(d)
    t = torch.empty(n, dtype=torch.int32, device="cuda")
    F = (1e-5 * rho0, -3e-6 * rho0, 1e-4) if forced else (0.0, 0.0, 0.0)
    torch.cuda.synchronize()
    assert probe.probe_pairs(int(elbm), int(forced), d.data_ptr(), n, rho0, tau, *F, a.data_ptr(),
                             b.data_ptr(), t.data_ptr()) == 0
    return a.cpu().numpy(), b.cpu().numpy(), t.cpu().numpy().astype(bool)


@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("rho0", [1.0, 0.3, 17.0])
def test_packed_bgk_equals_the_scalar_form(probe, rho0, forced):
    cells = np.concatenate([_cells(rho0, 0.05, 0.0, 5000, 1), _cells(rho0, 0.1, 0.02, 5001, 2)])
    a, b, _ = _pairs(probe, False, forced, cells, rho0)
    assert np.array_equal(a.view(np.uint32), b.view(np.uint32))


@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("rho0", [1.0, 0.3, 17.0])
def test_packed_entropic_equals_the_scalar_form(probe, rho0, forced):
    """Where the packed form takes a pair its bits are the scalar form's; it takes
    every pair within the series and none of those far beyond it."""
    near, edge, far = (_cells(rho0, 0.04, nz, 4001, 3 + k) for k, nz in enumerate((1e-3, 0.015, 0.2)))
    rest = np.zeros((64, 9), np.float32)
    mixed = near[:4000].copy()
    mixed[1::2] = far[:2000]
    nan = near[:64].copy()
    nan[::4, 3] = np.nan
    nan[1::4, 0] = np.inf
    for cells, takes in ((near, True), (edge, None), (far, False), (rest, True), (mixed, False),
                         (nan, None)):
        a, b, taken = _pairs(probe, True, forced, cells, rho0)
        if takes is not None:
            assert taken.all() if takes else taken.mean() < 0.01
        both = np.repeat(taken, 2)
        fin = both & np.isfinite(cells).all(1)
        assert np.array_equal(a[fin].view(np.uint32), b[fin].view(np.uint32))
        assert np.isnan(a[both & ~fin]).all()  # non-finite stays so
    _, _, taken = _pairs(probe, True, forced, edge, rho0)
    assert 0.0 < taken.mean() < 1.0
