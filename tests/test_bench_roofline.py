"""The benchmark's roofline of the row build is that of the form the library
took, whatever rate the time implies; the operations credited to the grid are
those of its plan (CPU only)."""
import numpy as np

import bench
from paper_2002_12471_gb300 import synthetic as S


def test_roofline_follows_the_form_of_the_build():
    ph, g, J, ns, ni = S.workload("dat64")
    args = dict(ph=ph, g=g, events=J, terms=1.1e11, terms_exact=1.5e11, ex2_peak=10068.0, ex2_basis="", pk=dict(bf16_tflops=1900.0),
                pk_kind="measured")
    # 15 ms imply 7.3e12 terms/s, less than the exponential unit forms: still the grid's
    grid = bench.build_roofline(True, ms=15.0, **args)
    assert grid["bound"] == "tensor" and grid["kernel"].startswith("k_grid_sum") and grid["equivalent_gterm_per_s"] < 10068.0
    path = bench.build_roofline(False, ms=15.0, **args)
    assert path["bound"] == "alu" and path["kernel"] == "k_pathsum"
    np.testing.assert_allclose([path["frac"], grid["frac"]],
                               [1.1e11 / 0.015 / 1e9 / 10068.0, bench.grid_sum_flops(ph, g) / 0.015 / 1e12 / 1900.0])


def test_grid_operations_are_the_plans():
    """64 x 64: no response reaches beyond 5.5 of the widest, and the products
    cannot need more than the 96 nodes of a window for each scatter pixel."""
    ph, g, *_ = S.workload("dat64")
    n_scat = int(np.count_nonzero(ph.mu))
    per_pair = bench.grid_sum_flops(ph, g) / (6.0 * g["n_angles"] * n_scat * n_scat)   # position x energy nodes
    assert 48 * 40 < per_pair < 96 * 64
