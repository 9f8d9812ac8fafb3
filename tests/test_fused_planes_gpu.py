"""The sensitivity's pass leaves the scatter planes of every angle behind
whenever they fit the table budget, whatever the number of scatter pixels: the
build then makes no tables.  At sizes on either side of the pieces that a block
holds at a time, sensitivity and rows are bit for bit those of the separate
kernels."""
import numpy as np
import pytest

from paper_2002_12471_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,full", [(64, True), (65, True), (128, False)])  # 4,096, 4,225 and 6,016 scatter pixels
def test_planes_of_large_objects_are_made_with_the_sensitivity(n, full):
    import torch

    import paper_2002_12471_gb300.lmosem as L
    ph = S.brain_phantom(n, 256.0 / n)
    if full:
        ph.mu[:] = np.maximum(ph.mu, 0.004)
    g = S.geometry(2, n, 256.0 / n, 200.0, angle0_rad=0.1)
    ev = S.simulate_events(ph, g, 90, seed=3)
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (ev.angle, ev.u_mm, ev.e_kev)]
    got = []
    for budget in (0, 1 << 20):
        ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=torch.cuda.current_stream(), profile=True,
                              table_budget_bytes=budget)
        try:
            nsup = L.lmosem_n_support(ctx)
            sens = torch.zeros((1, nsup), dtype=torch.float64, device=dev)
            L.lmosem_sensitivity(ctx, 1, sens)
            L.lmosem_profile_read(ctx)
            L.lmosem_build_model(ctx, *t, 1)
            tables = L.lmosem_profile_read(ctx)["wtable"][1]
            rows = torch.zeros((len(ev), nsup), dtype=torch.float32, device=dev)
            L.lmosem_model_rows(ctx, torch.arange(len(ev), device=dev), rows)
            got.append((tables, sens.cpu().numpy(), rows.cpu().numpy()))
        finally:
            L.lmosem_destroy(ctx)
    assert got[0][0] == 0 and got[1][0] > 0
    assert np.array_equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][2], got[1][2])
