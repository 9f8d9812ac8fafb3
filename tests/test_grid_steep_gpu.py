"""Rows of large event lists where the scatter sum falls steeply between the
grid's nodes: energies above every Compton energy that reaches a position from
a support smaller than the object, positions beyond the object when every
response is as narrow as the grid's step allows, positions between two objects.
The interpolation's error is small against the neighbouring grid values, not
against such a row, so these rows are summed path by path.  Every row against
the row built by itself: 2e-4 relative, plus of the row's largest entry 2e-6
for the path sum and, for the grid, 8 times 4e-7 (the stencil in energy, at a
row 1 / 8 of the values around it) and 3.6e-6 (the stencil in position), 1e-5
in all."""
import numpy as np
import pytest

from tests._helpers import gpu_reconstruct
from tests.test_grid_gpu import S

pytestmark = pytest.mark.gpu


def _disc(n, d, cx, cy, r):
    c = (np.arange(n) + 0.5 - 0.5 * n) * d
    x, y = np.meshgrid(c, c)
    return (x - cx) ** 2 + (y - cy) ** 2 <= r * r


def _problem(name):
    ph = S.brain_phantom(64, 4.0)
    g = S.geometry(4, 64, 4.0, 150.0, angle0_rad=0.2)
    if name == "brain support":
        return ph, g, ph.activity > 0.5
    if name == "striata":
        return ph, g, ph.activity > 2.0
    if name == "parallel responses":
        return ph, dict(g, coll_fwhm_slope=0.0, coll_fwhm0_mm=10.0), None
    mu = 0.0146 * (_disc(64, 4.0, -58, -5, 50) | _disc(64, 4.0, 58, 5, 50))
    return S.Phantom(mu=mu, activity=(mu > 0) * 1.0, pixel_mm=4.0), g, None


@pytest.mark.parametrize("name,on_grid", [("brain support", True), ("parallel responses", True), ("two objects", None),
                                          ("striata", None)])
def test_steep_rows(name, on_grid):
    ph, g, sup = _problem(name)
    per = 8000
    ev = S.simulate_events(ph, g, 4 * per, seed=17, batch=1 << 18)
    # 48 events far from the object in position or above it in energy
    yy, xx = np.nonzero(ph.mu > 0)
    X, Y = (xx + 0.5 - 32) * 4.0, (yy + 0.5 - 32) * 4.0
    k = np.arange(0, len(ev), len(ev) // 48)[:48]
    sig = (g["coll_fwhm0_mm"] + g["coll_fwhm_slope"] * g["radius_mm"]) / 2.3548
    for j, q in enumerate(k):
        th = g["angle0_rad"] + 2 * np.pi * ev.angle[q] / 4
        um = -X * np.sin(th) + Y * np.cos(th)
        ev.u_mm[q] = (um.max() if j & 1 else um.min()) + (1 if j & 1 else -1) * sig * (j % 12) / 4.2
        ev.e_kev[q] = (120.0, 145.0, 160.0, 172.0)[j // 12]
    if name == "two objects":
        ev.u_mm[k[:24]] = np.linspace(-9, 9, 24).astype(np.float32)
    rng = np.random.default_rng(0)
    pick = np.unique(np.concatenate([k, rng.choice(len(ev), 400, replace=False)]))
    got = gpu_reconstruct(ph, g, ev, 2, 1, rows=pick, support=sup)["rows"]
    sub = S.Events(ev.angle[pick], ev.u_mm[pick], ev.e_kev[pick], ev.order[pick])
    d = gpu_reconstruct(ph, g, sub, 2, 1, rows=np.arange(len(pick)), support=sup)["rows"]
    if on_grid is not None:
        assert np.array_equal(got, d) == (not on_grid)
    bound = 2e-4 * np.abs(d) + 1e-5 * d.max(axis=1, keepdims=True)
    bad = np.max(np.abs(got - d) / np.maximum(bound, 1e-300), axis=1)
    assert np.all(bad <= 1.0), (np.sum(bad > 1.0), bad.max())


def test_a_few_steep_rows_do_not_cost_a_second_build():
    """The shortest list that takes the grid (found within 3% of its length)
    still takes it with twenty steep rows, which are summed directly."""
    import torch

    import paper_2002_12471_gb300.lmosem as L
    ph, g, sup = _problem("parallel responses")
    ev = S.simulate_events(ph, g, 24000, seed=19, batch=1 << 18)
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (ev.angle, ev.u_mm, ev.e_kev)]
    ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, support=sup, stream=torch.cuda.current_stream())
    try:
        def on_grid(n, u, e):
            L.lmosem_build_model(ctx, t[0][:n], u[:n], e[:n], 1)
            return L.lmosem_model_on_grid(ctx)

        n = len(ev)
        assert on_grid(n, t[1], t[2])
        while on_grid(int(n / 1.03), t[1], t[2]):
            n = int(n / 1.03)
        u, e = t[1].clone(), t[2].clone()
        # 2.6 sigma beyond the object
        yy, xx = np.nonzero(ph.mu > 0)
        X, Y = (xx + 0.5 - 32) * 4.0, (yy + 0.5 - 32) * 4.0
        for q in range(1, 21):
            th = g["angle0_rad"] + 2 * np.pi * ev.angle[q] / 4
            u[q], e[q] = float((-X * np.sin(th) + Y * np.cos(th)).max()) + 11.0, 125.0
        assert on_grid(n, u, e)
        rows = torch.zeros((n, L.lmosem_n_support(ctx)), dtype=torch.float32, device=dev)
        L.lmosem_model_rows(ctx, torch.arange(n, device=dev), rows)
        got = rows[1:21].cpu().numpy().astype(np.float64)
    finally:
        L.lmosem_destroy(ctx)
    k = np.arange(1, 21)
    sub = S.Events(ev.angle[k], u[1:21].cpu().numpy(), e[1:21].cpu().numpy(), ev.order[k])
    d = gpu_reconstruct(ph, g, sub, 1, 0, rows=np.arange(20), support=sup)["rows"]
    bound = 2e-4 * np.abs(d) + 1e-5 * d.max(axis=1, keepdims=True)
    assert np.all(np.abs(got - d) <= bound), np.max(np.abs(got - d) / bound)
