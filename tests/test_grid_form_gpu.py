"""lmosem_model_on_grid reports the form of the last exact row build."""
import numpy as np
import pytest

from tests.test_grid_gpu import _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts,count,on_grid", [(dict(), None, True), (dict(), 100, False), (dict(e_sigma=-1.0), None, False)])
def test_form_of_the_last_build(opts, count, on_grid):
    import torch

    import paper_2002_12471_gb300.lmosem as L
    ph, g, ev, _ = _case(64, 3, 4000, seed=31)
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(np.ascontiguousarray(x[:count])).to(dev) for x in (ev.angle, ev.u_mm, ev.e_kev)]
    ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=torch.cuda.current_stream(), **opts)
    try:
        with pytest.raises(L.LmosemError) as ei:
            L.lmosem_model_on_grid(ctx)
        assert ei.value.status == L.EINVAL
        L.lmosem_build_model(ctx, *t, 1)
        assert L.lmosem_model_on_grid(ctx) is on_grid
    finally:
        L.lmosem_destroy(ctx)
