"""Large event lists take the grid only for the default cuts.  A caller that
asks for the exact sum (a negative e_sigma), or for more of the position
response than the default, gets every row path by path: bit for bit the row
built by itself, whose list is too short for the grid.  (With the energy cut
on, a row's bits do not depend on the list either.)"""
import numpy as np
import pytest

from tests._helpers import gpu_reconstruct
from tests.test_grid_gpu import S, _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts,on_grid", [(dict(), True), (dict(e_sigma=9.0), True), (dict(e_sigma=-1.0), False),
                                          (dict(k_sigma=8.0), False), (dict(k_sigma=20.0), False),
                                          (dict(e_sigma=5.0), False)])
def test_cuts_that_keep_the_path_sum(opts, on_grid):
    ph, g, ev, _ = _case(64, 3, 4000, seed=21)
    pick = np.arange(0, len(ev), 157)
    rows = gpu_reconstruct(ph, g, ev, 1, 1, rows=pick, **opts)["rows"]
    sub = S.Events(ev.angle[pick], ev.u_mm[pick], ev.e_kev[pick], ev.order[pick])
    alone = gpu_reconstruct(ph, g, sub, 1, 1, rows=np.arange(len(pick)), **opts)["rows"]
    assert np.array_equal(rows, alone) == (not on_grid)
