"""The binned model with energy bins that do not fill the kernel's groups of
three (1, 4, 5 and 8 bins) and a detector whose bins do not fill its tiles of
64 (41 and 70 bins): every row against the FP64 oracle, with the bound of the
model entries."""
import numpy as np
import pytest

from paper_2002_12471_gb300 import synthetic as S
from tests._helpers import oracle_problem, row_close
from tests.test_binned_gpu import gpu_binned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ebins,n_bins", [(1, 16), (4, 41), (5, 70), (8, 16)])
def test_energy_and_position_bins_outside_whole_groups(n_ebins, n_bins):
    ph, g, J, ns, ni = S.workload("tiny16")
    g = dict(g, n_angles=6, n_bins=n_bins, bin_mm=128.0 / n_bins)
    edges = np.linspace(100.0, 175.0, n_ebins + 1)
    rng = np.random.default_rng(n_ebins)
    counts = rng.poisson(0.7, (6, n_bins, n_ebins)).astype(np.float32)
    a, b, k = np.nonzero(counts > 0)
    p = oracle_problem(ph, g).model_binned(a, b, k, edges)
    out = gpu_binned(ph, g, counts, edges, 3, 1, rows=np.arange(len(a)))
    assert row_close(out["rows"], p) <= 1.0
