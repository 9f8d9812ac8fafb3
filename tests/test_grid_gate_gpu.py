"""The energy gate of the surrogate form on a large event list: the rows below
its cut are formed as a list of their events alone would be.  A few of them are
summed path by path, bit for bit, although the whole list is long enough for
the grid; when every row is below the cut they are the exact build's, bit for
bit, and the terms asked for afterwards are that build's."""
import numpy as np
import pytest

from tests._helpers import gpu_reconstruct
from tests.test_grid_gpu import S

pytestmark = pytest.mark.gpu


def test_gated_rows_take_the_form_of_their_own_list():
    import torch

    import paper_2002_12471_gb300.lmosem as L
    ph = S.brain_phantom(64, 4.0)
    g = S.geometry(3, 64, 4.0, 150.0, angle0_rad=0.2)
    ev = S.simulate_events(ph, g, 40000, seed=29, batch=1 << 18)
    # all but 60 of the events lie above 150 keV, none between 125 and 150
    high = np.flatnonzero(ev.e_kev > 150.0)
    low = np.flatnonzero(ev.e_kev < 125.0)[:60]
    k = np.sort(np.concatenate([high, low]))
    ev = S.Events(ev.angle[k], ev.u_mm[k], ev.e_kev[k], ev.order[k])
    low = ev.e_kev < 125.0
    # a network whose scatter is nothing: a row's error is the scatter's share of it
    params = [(np.zeros(s), np.zeros(s[0])) for s in ((256, 8), (256, 256), (256, 256), (256, 256), (1, 256))]
    blob = np.asarray(L.pack_surrogate(params), dtype=np.float32).copy()
    blob[-2:] = (-60.0, 1.0)
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (ev.angle, ev.u_mm, ev.e_kev)]

    def build(row_tol):
        ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=torch.cuda.current_stream())
        try:
            nsup = L.lmosem_n_support(ctx)
            L.lmosem_surrogate_load(ctx, torch.from_numpy(blob).to(dev))
            L.lmosem_set_surrogate_check(ctx, 1e6, len(ev))
            L.lmosem_set_surrogate_gate(ctx, row_tol)
            L.lmosem_build_model(ctx, *t, 1, "surrogate")
            buf = torch.zeros((len(ev), nsup), dtype=torch.float32, device=dev)
            L.lmosem_model_rows(ctx, torch.arange(len(ev), device=dev), buf)
            return buf.cpu().numpy().astype(np.float64), L.lmosem_surrogate_gate(ctx), L.lmosem_model_terms(ctx)
        finally:
            L.lmosem_destroy(ctx)

    exact = gpu_reconstruct(ph, g, ev, 1, 0, rows=np.arange(len(ev)))
    sub = S.Events(ev.angle[low], ev.u_mm[low], ev.e_kev[low], ev.order[low])
    alone = gpu_reconstruct(ph, g, sub, 1, 0, rows=np.arange(int(low.sum())))
    assert not np.array_equal(exact["rows"][low], alone["rows"])   # the whole list takes the grid
    rows, (cut, frac), terms = build(0.9)
    assert 125.0 <= cut <= 150.0 and frac == low.mean(), (cut, frac)
    assert np.array_equal(rows[low], alone["rows"])
    assert terms == alone["terms"]
    rows, (cut, frac), terms = build(1e-9)
    assert frac == 1.0
    assert np.array_equal(rows, exact["rows"])
    assert terms == exact["terms"]
