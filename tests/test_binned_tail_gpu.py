"""Binned rows that do not fill the pass's last group of rows: a row past the
end has no weight, whatever the memory after the weights holds (device memory
is reused, and the row map's empty entries are NaN when read as floats)."""
import numpy as np
import pytest

from paper_2002_12471_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
@pytest.mark.parametrize("n_rows", [1, 37, 38, 39, 40])
def test_rows_past_the_end_weigh_nothing(variant, n_rows):
    import torch

    import paper_2002_12471_gb300.lmosem as L
    ph, g, J, ns, ni = S.workload("tiny16")
    g = dict(g, n_angles=6)
    counts = np.zeros((6, g["n_bins"], 1), np.float32)
    # detector bins over the object, filled from the first angle on
    at = [(a, b) for a in range(6) for b in range(g["n_bins"] // 4, g["n_bins"] - g["n_bins"] // 4)][:n_rows]
    assert len(at) == n_rows
    for k, (a, b) in enumerate(at):
        counts[a, b, 0] = 1.0 + k % 5
    d_counts = torch.from_numpy(counts).cuda()
    first = None
    for _ in range(4):
        ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=torch.cuda.current_stream(), pass_variant=variant)
        try:
            nsup = L.lmosem_n_support(ctx)
            sens = torch.zeros((1, nsup), dtype=torch.float64, device="cuda")
            L.lmosem_sensitivity(ctx, 1, sens)
            f = torch.empty(nsup, device="cuda")
            for _ in range(2):
                L.lmosem_build_model_binned(ctx, d_counts, (100.0, 175.0), 1)
                L.lmosem_init_image(ctx, 1.0, f)
                f0 = f.cpu().numpy().astype(np.float64)
                rows = torch.empty((n_rows, nsup), device="cuda")
                L.lmosem_model_rows(ctx, torch.arange(n_rows, device="cuda"), rows)
                L.lmosem_iterate(ctx, 1, 1.0, f)
                p = rows.cpu().numpy().astype(np.float64)
                got = f.cpu().numpy().astype(np.float64)
                assert np.isfinite(got).all()
                w = counts[tuple(np.transpose([(a, b, 0) for a, b in at]))].astype(np.float64)
                want = f0 / sens.cpu().numpy()[0] * (p.T @ (w / (p @ f0)))
                assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
                assert first is None or np.array_equal(got, first)
                first = got
        finally:
            L.lmosem_destroy(ctx)
