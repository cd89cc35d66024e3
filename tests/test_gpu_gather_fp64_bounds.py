"""The FP64 gather on cells whose terms lie close to their fixed-point bounds (beams, uniform
cubes, shells of one speed), by a warp a cell (few cells) and by eight lanes (many)."""

import numpy as np
import pytest

from test_fixed_point_lanes_host import near_bounds
from test_gpu_gather_fp64 import _check

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KINDS = ["beams below", "beams above", "beams low", "beams across", "cube", "shell"]


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("n_cells", [1, 5, 64, 2500])
def test_terms_near_their_bounds(n_cells, dtype):
    """1e-14 as for the plain cells: some ten FP64 roundings of each side."""
    rng = np.random.default_rng(n_cells)
    sizes = [300, 1000, 5000] if n_cells <= 64 else [300, 257, 960]
    cells = [near_bounds(KINDS[(c + c // 6) % 6], sizes[c % 3], rng) for c in range(max(n_cells, 6))]
    if n_cells == 1:
        for x in cells:
            _check(x.astype(dtype), np.array([0, x.shape[1]]), 1e-14)
        return
    cells = cells[:n_cells]
    off = np.concatenate([[0], np.cumsum([x.shape[1] for x in cells])]).astype(np.int64)
    _check(np.concatenate(cells, axis=1).astype(dtype), off, 1e-14)
