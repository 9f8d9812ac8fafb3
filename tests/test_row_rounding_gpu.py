"""Scaled rows (FP16, BF16) are the FP32 rows divided by their scale, rounded to
nearest and multiplied by it again, bit for bit, at row widths on either side of
the rounding kernel's two block sizes and beyond the columns a block holds in
registers."""
import numpy as np
import pytest

from paper_2002_12471_gb300 import synthetic as S
from tests._helpers import gpu_reconstruct

pytestmark = pytest.mark.gpu


def _bf16(x):
    b = x.view(np.uint32).astype(np.uint64)
    return ((b + 0x7FFF + ((b >> 16) & 1)) >> 16 << 16).astype(np.uint32).view(np.float32)


@pytest.mark.parametrize("n", [17, 45, 46, 91])  # 289, 2,025, 2,116 and 8,281 columns
def test_rounded_rows(n):
    ph = S.brain_phantom(n, 256.0 / n)
    ph.mu[:] = np.maximum(ph.mu, 0.005)  # every pixel is support
    g = S.geometry(2, n, 256.0 / n, 200.0, angle0_rad=0.1)
    ev = S.simulate_events(ph, g, 37, seed=3)

    def rows(fmt, support=None):  # without the energy cut, whose column tiles depend on the support
        out = gpu_reconstruct(ph, g, ev, 1, 1, fmt, support=support, rows=np.arange(len(ev)), e_sigma=-1.0)
        return out["rows"].astype(np.float32)

    first = np.arange(n * n).reshape(n, n) < n * n // 2  # FP32 passes end at 8,192 columns: two halves
    h = np.concatenate([rows("fp32", first), rows("fp32", ~first)], axis=1) if n * n > 8192 else rows("fp32")
    assert h.shape == (len(ev), n * n)
    top = h.max(axis=1, keepdims=True)
    c = top / np.float32(32768.0)
    assert np.array_equal(rows("fp16"), (h * (np.float32(1.0) / c)).astype(np.float16).astype(np.float32) * c)
    assert np.array_equal(rows("bf16"), _bf16(h * (np.float32(1.0) / top)) * top)
