"""The bounded waits of the scatter sum on the grid take the context's budget:
a one-cycle budget makes the model build of a large event list return ETIMEOUT
and leaves no model behind; with the budget restored the same context builds
the rows of a fresh context bit for bit."""
import numpy as np
import pytest

from tests._helpers import gpu_reconstruct
from tests.test_grid_gpu import _case, _direct

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", ["fp32", "fp16"])
def test_grid_wait_budget_runs_out_cleanly(fmt):
    import torch

    import paper_2002_12471_gb300.lmosem as L
    ph, g, ev, _ = _case(64, 3, 4000, seed=9)
    pick = np.arange(0, len(ev), 131)
    ref = gpu_reconstruct(ph, g, ev, 1, 1, fmt, rows=pick)["rows"]
    assert not np.array_equal(ref, _direct(ph, g, ev, pick, 1, fmt)["rows"])   # the grid was used
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (ev.angle, ev.u_mm, ev.e_kev)]
    ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=torch.cuda.current_stream(), wait_budget_cycles=1)
    try:
        for _ in range(2):
            with pytest.raises(L.LmosemError) as ei:
                L.lmosem_build_model(ctx, *t, 1, fmt)
            assert ei.value.status == L.ETIMEOUT
            assert L.lmosem_model_bytes(ctx) == 0
        L.lmosem_set_wait_budget(ctx, 0)
        L.lmosem_build_model(ctx, *t, 1, fmt)
        buf = torch.zeros((len(pick), L.lmosem_n_support(ctx)), dtype=torch.float32, device=dev)
        L.lmosem_model_rows(ctx, torch.as_tensor(pick, device=dev), buf)
        assert np.array_equal(buf.cpu().numpy().astype(np.float64), ref)
    finally:
        L.lmosem_destroy(ctx)
