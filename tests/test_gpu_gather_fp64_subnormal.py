"""The FP64 gather of FP32 velocities so small that some are FP32 subnormals."""

import numpy as np
import pytest

from test_gpu_gather_fp64 import _check, _population

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells", [5, 3000])
@pytest.mark.parametrize("exponent", [-130, -124, -118, -100, -70, -60])
def test_fp32_subnormals(exponent, n_cells):
    """1e-14 as for velocities of order one: an FP32 subnormal is an exact FP64 number."""
    v, off = _population([12 + 7 * (c % 11) for c in range(n_cells)], (1.0, 1.7, 0.6), 3)
    v = (v * 2.0**exponent).astype(np.float32)
    if exponent <= -118 and n_cells == 3000:
        assert ((v != 0) & (np.abs(v) < 2.0**-126)).any()
    _check(v, off, 1e-14)
