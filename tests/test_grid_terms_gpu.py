"""The path terms of a build on the grid are counted when they are asked for and
not before: a build of binned rows (or of another list that is refused) on the
same context does no work for them, and the count can still be asked for
afterwards.  It is that of the path sum, which adds up over lists short enough
for it."""
import numpy as np
import pytest

from tests._helpers import gpu_reconstruct
from tests.test_grid_gpu import S, _case

pytestmark = pytest.mark.gpu


def test_terms_are_counted_on_request_only():
    import torch

    import paper_2002_12471_gb300.lmosem as L
    ph, g, ev, _ = _case(64, 3, 3000, seed=23)
    parts = 0
    for k in range(0, len(ev), 450):
        sub = S.Events(ev.angle[k:k + 450], ev.u_mm[k:k + 450], ev.e_kev[k:k + 450], ev.order[k:k + 450])
        parts += gpu_reconstruct(ph, g, sub, 1, 0)["terms"]
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (ev.angle, ev.u_mm, ev.e_kev)]
    edges = np.linspace(100.0, 175.0, 3)
    counts = torch.ones((3, 64, 2), dtype=torch.float32, device=dev)
    launches, seen = {}, {}
    for first in ("events", "none"):
        ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=torch.cuda.current_stream())
        try:
            if first == "events":
                L.lmosem_build_model(ctx, *t, 1)
                bad = t[1].clone()
                bad[7] = 1e6
                with pytest.raises(L.LmosemError) as ei:   # releases the model
                    L.lmosem_build_model(ctx, t[0], bad, t[2], 1)
                assert ei.value.status == L.EINVAL
            else:   # what the pass needs once per context
                L.lmosem_build_model(ctx, *(x[:60] for x in t), 1)
            n0 = L.lmosem_launch_count(ctx)
            L.lmosem_build_model_binned(ctx, counts, edges, 1)
            launches[first] = L.lmosem_launch_count(ctx) - n0
            seen[first] = (L.lmosem_model_terms(ctx), L.lmosem_model_terms(ctx))
        finally:
            L.lmosem_destroy(ctx)
    assert launches["events"] == launches["none"]
    assert seen["events"] == (parts, parts)
