"""Events outside the grid's region are summed directly, each counted as 30 rows
of the path sum: a list that the grid wins by little keeps the path sum when
0.6% of its events lie there, one that it wins by far still takes the grid."""
import numpy as np
import pytest

from tests._helpers import gpu_reconstruct
from tests.test_grid_gpu import S

pytestmark = pytest.mark.gpu


def _on_grid(ph, g, ev, outside):
    u = ev.u_mm.copy()
    u[::167] = 127.0 if outside else u[::167]
    pick = np.arange(1, len(ev), max(1, len(ev) // 40))
    lists = [S.Events(x.angle, w, x.e_kev, x.order) for x, w in
             ((ev, u), (S.Events(ev.angle[pick], None, ev.e_kev[pick], ev.order[pick]), u[pick]))]
    a = gpu_reconstruct(ph, g, lists[0], 1, 0, rows=pick)["rows"]
    b = gpu_reconstruct(ph, g, lists[1], 1, 0, rows=np.arange(len(pick)))["rows"]
    return not np.array_equal(a, b)   # a path-sum row does not depend on the list


def test_outside_events_count_at_their_cost():
    ph = S.brain_phantom(64, 4.0)
    g = S.geometry(3, 64, 4.0, 150.0, angle0_rad=0.2)
    full = S.simulate_events(ph, g, 24000, seed=5, batch=1 << 18)

    def first(n):
        return S.Events(full.angle[:n], full.u_mm[:n], full.e_kev[:n], full.order[:n])

    assert _on_grid(ph, g, full, True)
    n = len(full)
    while _on_grid(ph, g, first(int(n / 1.03)), False):
        n = int(n / 1.03)
    assert 300 < n < len(full)             # the shortest list on the grid, within 3%
    assert not _on_grid(ph, g, first(n), True)
