"""Model rows of large event lists: the scatter sum on a grid of positions and
energies, interpolated at the events (csrc/grid.cu).  It is chosen when an
angle holds many events, so these cases have few angles.  Rows against the
FP64 oracle with the bound of every model entry (2e-4 relative plus 2e-6 of
the row maximum; the grid's own error is below 1e-6 of the row maximum:
interpolation 2e-7, FP16-split products 2e-8, truncated tensor-core sums 4e-7),
including events far outside the object and grids that do not divide the
kernels' tiles."""
import numpy as np
import pytest

import oracle
from tests._helpers import gpu_reconstruct, oracle_problem
from paper_2002_12471_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def _case(n, angles, per_angle, seed):
    ph = S.brain_phantom(n, 256.0 / n)
    g = S.geometry(angles, n, 256.0 / n, 150.0, angle0_rad=0.2)
    ev = S.simulate_events(ph, g, angles * per_angle, seed=seed, batch=1 << 18)
    half = 0.5 * n * ph.pixel_mm
    # a few events that no photon of the object would give: edges of the
    # detector and of the window (they are summed path by path)
    k = np.arange(0, len(ev), max(1, len(ev) // 24))[:24]
    ev.u_mm[k[:12]] = np.linspace(-half, half, 12).astype(np.float32)
    ev.e_kev[k[12:]] = np.linspace(100.0, 175.0, 12).astype(np.float32)
    return ph, g, ev, k


def _direct(ph, g, ev, pick, ns, fmt="fp32"):
    """The rows of a few events built by themselves: path by path."""
    sub = S.Events(ev.angle[pick], ev.u_mm[pick], ev.e_kev[pick], ev.order[pick])
    return gpu_reconstruct(ph, g, sub, ns, 1, fmt, rows=np.arange(len(pick)))


@pytest.mark.parametrize("n,angles,per_angle", [(64, 3, 4000), (61, 2, 5003), (100, 3, 2048)])
def test_grid_rows_against_oracle_and_path_sum(n, angles, per_angle):
    ph, g, ev, special = _case(n, angles, per_angle, seed=7)
    rng = np.random.default_rng(0)
    pick = np.unique(np.concatenate([special, rng.choice(len(ev), 60, replace=False)]))
    out = gpu_reconstruct(ph, g, ev, 1, 1, rows=pick)
    d = _direct(ph, g, ev, pick, 1)["rows"]
    assert not np.array_equal(out["rows"], d)   # the grid was used
    # every row against the path sum's; far outside the object both leave out
    # what lies beyond 6 sigma, so only the others are compared with the oracle
    bound = 2e-4 * np.abs(d) + 2e-6 * d.max(axis=1, keepdims=True)
    assert np.all(np.abs(out["rows"] - d) <= bound), np.max(np.abs(out["rows"] - d) / bound)
    inner = np.setdiff1d(np.arange(len(pick)), np.searchsorted(pick, special))
    at = pick[inner]
    P = oracle_problem(ph, g)
    p = P.model(ev.angle[at], ev.u_mm[at], ev.e_kev[at])
    bound = 2e-4 * np.abs(p) + 2e-6 * p.max(axis=1, keepdims=True)
    got = out["rows"][inner]
    assert np.all(np.abs(got - p) <= bound), np.max(np.abs(got - p) / bound)
    err, ref = (np.linalg.norm(x - p) / np.linalg.norm(p) for x in (got, d[inner]))
    assert err <= max(1e-6, 1.5 * ref), (err, ref)


def test_grid_groups_formats_and_terms():
    """Angle groups of one (a small table budget) give the bits of one group;
    scaled formats round the same rows; two builds are bitwise equal; the
    term count is that of the path sum (additive over events)."""
    ph, g, ev, _ = _case(64, 4, 3001, seed=11)
    pick = np.arange(0, len(ev), 97)
    a = gpu_reconstruct(ph, g, ev, 2, 2, rows=pick)
    b = gpu_reconstruct(ph, g, ev, 2, 2, rows=pick, table_budget_bytes=1 << 20)
    c = gpu_reconstruct(ph, g, ev, 2, 2, rows=pick)
    for k in ("rows", "f", "sens"):
        assert np.array_equal(a[k], b[k]) and np.array_equal(a[k], c[k]), k
    for fmt, unit in (("fp16", 2.0 ** -11), ("bf16", 2.0 ** -8)):
        h = gpu_reconstruct(ph, g, ev, 2, 2, fmt, rows=pick)
        tol = 1.01 * unit * a["rows"] + 2.0 ** -24 * a["rows"].max(axis=1, keepdims=True)
        assert np.all(np.abs(h["rows"] - a["rows"]) <= tol)
    parts = 0
    for k in range(0, len(ev), 400):
        sub = S.Events(ev.angle[k:k + 400], ev.u_mm[k:k + 400], ev.e_kev[k:k + 400], ev.order[k:k + 400])
        parts += gpu_reconstruct(ph, g, sub, 2, 1)["terms"]
    assert a["terms"] == parts


def test_grid_batch_matches_single_sets():
    """Realisations of one batch share the grid: every image within 1e-5 of
    its single-set reconstruction."""
    import torch

    import paper_2002_12471_gb300.lmosem as L
    ph, g, ev, _ = _case(64, 3, 6000, seed=5)
    off = np.array([0, 7000, 7000, 11000, len(ev)], dtype=np.int64)
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (ev.angle, ev.u_mm, ev.e_kev)]
    ctx = L.lmosem_create(ph.mu, ph.pixel_mm, g, stream=torch.cuda.current_stream())
    try:
        L.lmosem_sensitivity(ctx, 1)
        L.lmosem_build_model_batch(ctx, *t, off, 1)
        f = torch.zeros((4, L.lmosem_n_support(ctx)), dtype=torch.float32, device=dev)
        L.lmosem_init_image_batch(ctx, 1.0, f)
        L.lmosem_iterate_batch(ctx, 3, 1.0, f)
        got = f.cpu().numpy().astype(np.float64)
    finally:
        L.lmosem_destroy(ctx)
    for r in (0, 2, 3):
        s = slice(off[r], off[r + 1])
        one = gpu_reconstruct(ph, g, S.Events(ev.angle[s], ev.u_mm[s], ev.e_kev[s], ev.order[s]), 1, 3)
        assert oracle.rel_l2(got[r], one["f"]) <= 1e-5, r


def test_grid_not_used_where_its_premises_fail():
    """A position cut below the default leaves steps in the sum, and too many
    events outside the object cost more than the grid saves: both keep the
    path sum, whose rows do not depend on the other events."""
    ph, g, ev, _ = _case(64, 2, 4000, seed=3)
    pick = np.arange(0, len(ev), 211)
    cut = gpu_reconstruct(ph, g, ev, 1, 1, rows=pick, k_sigma=4.0)["rows"]
    sub = S.Events(ev.angle[pick], ev.u_mm[pick], ev.e_kev[pick], ev.order[pick])
    assert np.array_equal(cut, gpu_reconstruct(ph, g, sub, 1, 1, rows=np.arange(len(pick)), k_sigma=4.0)["rows"])
    ev.u_mm[::50] = 127.0
    out = gpu_reconstruct(ph, g, ev, 1, 1, rows=pick)["rows"]
    assert np.array_equal(out, _direct(ph, g, ev, pick, 1)["rows"])
