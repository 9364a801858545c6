"""The launch shape does not enter the results: every rows-per-warp and
projection setting of the batched FP32 kernel, in both storages, leaves the
same populations bit for bit, for the collisions whose arithmetic does not
depend on the kernel variant (BGK and the entropic one).  The damping of the
paper's forcing is the part that sums over cells: heights that leave ragged last
groups of rows, one group and several, a second column of four cells."""
import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu

GRIDS = [(128, 40), (256, 200), (132, 100), (4, 6), (640, 64), (64, 129)]


@pytest.fixture(scope="module")
def P():
    import paper_1809_06735_gb300 as P
    return P


def _run(P, collision, storage, rows, proj_rows, graph=0):
    members = [P.Member(nx, ny, 0.52 + 0.01 * i, 1.0, 2, 4, 1e-4, 1e-4, 0.0, 1e-2, collision)
               for i, (nx, ny) in enumerate(GRIDS)]
    lat = P.Lattice(members, precision=32, storage=storage, diag_every=9, graph_steps=graph)
    lat.set_launch(4, rows, 0, proj_rows)
    for m, (nx, ny) in enumerate(GRIDS):
        f = [li.smooth_fields(nx, ny, 3 * m + k, amp=a) for k, a in enumerate((.01, .03, .03))]
        lat.init_fields(m, 1.0 + f[0], f[1], f[2])
    lat.step(9)
    out = [lat.get_populations_host(m) for m in range(len(GRIDS))]
    stats = lat.subvolume_balance_batch(list(range(3)), [3, 16])
    lat.close()
    return out, stats


@pytest.mark.parametrize("collision", [0, 3])
def test_damping_does_not_depend_on_the_launch(P, collision):
    want, stats = _run(P, collision, 1, 2, 8)
    for storage in (1, 2):
        for rows, proj_rows in ((1, 8), (2, 1), (2, 4), (2, 13), (4, 16), (1, 24), (2, 64)):
            got, st = _run(P, collision, storage, rows, proj_rows, graph=4 if rows == 4 else 0)
            for m, (a, b) in enumerate(zip(got, want)):
                assert np.array_equal(a, b), (storage, rows, proj_rows, GRIDS[m])
            assert np.array_equal(st, stats), (storage, rows, proj_rows)
