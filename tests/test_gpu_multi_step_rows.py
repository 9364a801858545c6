"""Blocks of more rows than the grid has, up to the largest number of the C
interface, are whole columns: accepted, and the same populations bit for bit."""
import numpy as np
import pytest

import lbm_inputs as li

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [64, 65, 513, 2 ** 31 - 512, 2 ** 31 - 1])
def test_rows_above_the_grid(rows):
    import paper_1809_06735_gb300 as P
    out = []
    for steps, r in ((1, 64), (3, rows)):
        lat = P.Lattice([P.Member(132, 64, 0.56), P.Member(8, 512, 0.6)], precision=32, storage=2)
        lat.set_steps_per_launch(steps, r)
        assert lat.steps_per_launch == steps
        for m, (nx, ny) in enumerate(((132, 64), (8, 512))):
            lat.set_populations(m, li.random_populations(nx, ny, seed=m, rel_noise=0.03))
        lat.step(7)
        out.append([lat.get_populations_host(m) for m in range(2)])
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
