"""The balancing errors of a symmetric flow stepped in fixed point.  A Taylor-Green
vortex's errors are small differences of the balance's terms, so they show the
rounding of the state: the time derivative of E = u^2 / 2 over three levels, 4 u0
times the velocities' error (some 1e-16 after 100 steps), against terms of
2 nu rho S^2 ~ 0.03 (2 pi u0 / n)^2, i.e. 1e-8 (n / 256)^2 at u0 = 0.01.  The
reference (tests/golden/taylor_green_fp64.json) is the oracle's source compiled
with long double (64-bit significands), run from the same populations; running
this file writes it anew where long double is that type.

Measured: 192^2 8e-10 to 1.1e-9, 256^2 3.9e-9 to 4.7e-9; the FP64 form of the step
6e-9 to 8e-9 and 1.3e-8 to 1.7e-8 (populations 7e-16 off against 1.5e-14)."""
import json
import os

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
GOLDEN = os.path.join(HERE, "golden", "taylor_green_fp64.json")
TAU, STEPS, LS, GRIDS = 0.6, 100, [4, 8, 16, 32], (192, 256)


def _start(n, orc):
    """Populations of the vortex, the same bits on every machine."""
    s, c = (np.round(f(2.0 * np.pi * (np.arange(n) + 0.37) / n) * 2.0 ** 40) / 2.0 ** 40
            for f in (np.sin, np.cos))
    u0, k = 0.01, np.ones((n, n))
    rho = 1.0 - 0.75 * u0 * u0 * ((2.0 * c * c - 1.0)[None, :] + (2.0 * c * c - 1.0)[:, None])
    return orc.init(rho, u0 * s[None, :] * c[:, None] * k, -u0 * c[None, :] * s[:, None] * k)


@pytest.mark.gpu
@pytest.mark.parametrize("n", GRIDS)
def test_balancing_errors(orc, n):
    import paper_1809_06735_gb300 as P
    with open(GOLDEN) as fh:
        want = np.array(json.load(fh)[str(n)])
    lat = P.Lattice([P.Member(n, n, TAU)], precision=64, diag_every=STEPS)
    lat.set_populations(0, _start(n, orc))
    lat.step(STEPS)
    got = lat.subvolume_balance(0, LS)[:, :2]
    lat.close()
    assert np.linalg.norm(got - want) / np.linalg.norm(want) < 1e-8 * (n / 256.0) ** 2


def _write_golden():
    import ctypes
    import re
    import subprocess
    import sys
    import tempfile
    sys.path.insert(0, os.path.dirname(HERE))
    import oracle as orc
    ld, P, I, D = np.longdouble, ctypes.c_void_p, ctypes.c_int, ctypes.c_longdouble
    assert np.finfo(ld).nmant == 63, "the reference needs x87 long doubles"
    with open(os.path.join(os.path.dirname(HERE), "oracle", "lbm_oracle.c")) as fh:
        src = re.sub(r"/\*.*?\*/", "", fh.read(), flags=re.S)
    src = re.sub(r"\bdouble\b", "long double", src).replace("<math.h>", "<tgmath.h>")
    src = re.sub(r"(?<![\w.])(\d+\.\d*(?:[eE][-+]?\d+)?|\d+[eE][-+]?\d+)(?![\w.])", r"\1L", src)
    with tempfile.TemporaryDirectory() as d:
        with open(os.path.join(d, "ld.c"), "w") as fh:
            fh.write(src)
        subprocess.run(["gcc", "-O2", "-fPIC", "-shared", "-std=c99", "-ffp-contract=off", "-o",
                        d + "/ld.so", d + "/ld.c", "-lm"], check=True)
        lib = ctypes.CDLL(d + "/ld.so")

    class Model(ctypes.Structure):
        _fields_ = [("kind", I), ("F0", D), ("kf", I), ("alpha", D), ("phase", D), ("FR0", D),
                    ("collision", I), ("Cs", D)]

    lib.orc_run.argtypes = [I, I, D, P, P, I]
    lib.orc_terms_from_populations.argtypes = [I, I, D, P, P, P, P, P]
    lib.orc_balance_stats.argtypes = [I, I, P, P, I, P, I, P, P]
    out, m, L = {}, Model(), np.asarray(LS, np.int32)
    for n in GRIDS:
        f, level = np.ascontiguousarray(_start(n, orc), ld), []
        for k in (STEPS - 2, 1, 1):
            lib.orc_run(n, n, ld(TAU), ctypes.byref(m), f.ctypes.data, k)
            level.insert(0, f.copy())
        T, st = np.zeros((13, n, n), ld), np.zeros((len(LS), 15, 2), ld)
        lib.orc_terms_from_populations(n, n, ld(TAU), ctypes.byref(m), *[a.ctypes.data for a in level],
                                       T.ctypes.data)
        lib.orc_balance_stats(n, n, T.ctypes.data, L.ctypes.data, len(LS), None, n * n,
                              st.ctypes.data, None)
        out[str(n)] = st[:, :2].astype(float).tolist()
    with open(GOLDEN, "w") as fh:
        json.dump(out, fh, indent=1)


if __name__ == "__main__":
    _write_golden()
