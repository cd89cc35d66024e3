"""The adjoint's FP32 particle pass with moment gradients below FP32's normal range: large
velocities (order 1e4) make normal gradients of them."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells", [300, 32768 + 77])
def test_subnormal_moment_gradients(n_cells):
    """Within 3e-5 of the cell's largest gradient for the FP32 roundings (as for gradients
    of order one) and 2^-150 / 4e-41 = 2e-5 for each of some five coefficients that are
    rounded to FP32 subnormals (1e-38 / 4 at least, divided by up to 50 particles)."""
    from paper_2606_15622_gb300 import api
    rng = np.random.default_rng(n_cells)
    counts = np.array([(8, 13, 21, 50)[c % 4] for c in range(n_cells)])
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    n = int(off[-1])
    v = torch.from_numpy((1e4 * rng.standard_normal((3, n))).astype(np.float32)).cuda()
    offd = torch.from_numpy(off).cuda()
    tau = torch.ones(n_cells, dtype=torch.float64, device="cuda")
    mom = api.fp_moments(v.double(), offd, prec="fp64")
    y = torch.zeros((n_cells, 9), dtype=torch.float64, device="cuda")
    fl = torch.full((n_cells,), api.FLAG_FEW, dtype=torch.int32, device="cuda")  # the closure's own part is zero
    gm = torch.zeros((n_cells, 30), dtype=torch.float64, device="cuda")
    gm[:, 27:] = torch.from_numpy(rng.uniform(0.25, 1.0, (n_cells, 3)) * 1e-38).cuda()
    _, g32 = api.fp_closure_backward(v, offd, tau, mom, y, fl, y, grad_moments_in=gm)
    _, g64 = api.fp_closure_backward(v.double(), offd, tau, mom, y, fl, y, grad_moments_in=gm)
    cell = torch.repeat_interleave(torch.arange(n_cells, device="cuda"), torch.from_numpy(counts).cuda())
    top = torch.zeros(n_cells, dtype=torch.float64, device="cuda")
    top.scatter_reduce_(0, cell, g64.abs().max(dim=0).values, "amax")
    assert (top > 1e-30).all()
    err = (g32.double() - g64).abs().max(dim=0).values
    assert (err <= 1.3e-4 * top[cell]).all()
