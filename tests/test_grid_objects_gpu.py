"""Rows on the grid against the FP64 oracle for the 128 x 128 brain (the form
that the largest workload takes) and for maps whose path weights span many
orders of magnitude, where the 16-bit parts of the products have the least
room: a lead insert (2 / mm), one pixel of 20 / mm, and ten times the brain's
attenuation.  The bound of every model entry (2e-4 relative plus 2e-6 of the
row's maximum), and no larger an error than the path sum's by more than half,
or 1e-6, in relative L2."""
import numpy as np
import pytest

from tests._helpers import gpu_reconstruct, oracle_problem, row_close
from tests.test_grid_gpu import S

pytestmark = pytest.mark.gpu


def _map(name):
    ph = S.brain_phantom(128 if name == "brain 128" else 64, 2.0 if name == "brain 128" else 4.0)
    if name == "lead":
        ph.mu[20:23, 40:43] = 2.0
    elif name == "one pixel":
        ph.mu[31, 31] = 20.0
    elif name == "ten times":
        ph.mu[:] *= 10.0
    return ph


@pytest.mark.parametrize("name,per_angle", [("brain 128", 2000), ("lead", 4000), ("one pixel", 4000), ("ten times", 4000)])
def test_grid_rows_against_oracle(name, per_angle):
    ph, source = _map(name), _map("brain 128" if name == "brain 128" else "brain")
    n = ph.mu.shape[0]
    g = S.geometry(2, n, 256.0 / n, 150.0, angle0_rad=0.2)
    ev = S.simulate_events(source, g, 2 * per_angle, seed=41, batch=1 << 18)   # photons of the plain map
    pick = np.sort(np.random.default_rng(1).choice(len(ev), 80, replace=False))
    got = gpu_reconstruct(ph, g, ev, 1, 0, rows=pick)["rows"]
    sub = S.Events(ev.angle[pick], ev.u_mm[pick], ev.e_kev[pick], ev.order[pick])
    path = gpu_reconstruct(ph, g, sub, 1, 0, rows=np.arange(len(pick)))["rows"]
    assert not np.array_equal(got, path)   # the grid was used
    p = oracle_problem(ph, g).model(ev.angle[pick], ev.u_mm[pick], ev.e_kev[pick])
    assert row_close(got, p) <= 1.0
    err, ref = (np.linalg.norm(x - p) / np.linalg.norm(p) for x in (got, path))
    assert err <= max(1e-6, 1.5 * ref), (err, ref)
