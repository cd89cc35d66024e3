"""The adjoint's FP32 particle pass beyond the group kernel's cell count (tables of up to 32
cells a warp, shares that cut cells, quads that cross them, every alignment of the three
component arrays) against the FP64 pass on the same velocities."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra", [0, 1, 2, 3])
@pytest.mark.parametrize("sizes", [[8, 13, 0, 21, 1, 40, 9], [2, 3, 5, 4], [100, 2, 900, 30]])
def test_fp32_pass_against_fp64(extra, sizes):
    """Within 3e-5 of the cell's largest gradient: some 60 FP32 roundings of terms up to a
    few times it.  (The moment gradients are the call's own input, so that both passes
    read the same ones; one particle's worth of cells carry large ones.)"""
    from paper_2606_15622_gb300 import api
    n_cells = 32768 + 233
    rng = np.random.default_rng(extra + 10 * len(sizes))
    counts = np.array([sizes[c % len(sizes)] for c in range(n_cells)])
    counts[-1] += (extra - counts.sum()) % 4  # component arrays at every offset from 16 bytes
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    n = int(off[-1])
    assert n % 4 == extra
    v = torch.from_numpy((rng.standard_normal((3, n)) + np.array([[0.5], [-0.3], [0.0]])).astype(np.float32)).cuda()
    offd = torch.from_numpy(off).cuda()
    tau = torch.ones(n_cells, dtype=torch.float64, device="cuda")
    mom = api.fp_moments(v.double(), offd, prec="fp64")
    y = torch.zeros((n_cells, 9), dtype=torch.float64, device="cuda")
    fl = torch.full((n_cells,), api.FLAG_FEW, dtype=torch.int32, device="cuda")  # the closure's own part is zero
    gm = torch.from_numpy(rng.standard_normal((n_cells, 30))).cuda()
    _, g32 = api.fp_closure_backward(v, offd, tau, mom, y, fl, y, grad_moments_in=gm)
    _, g64 = api.fp_closure_backward(v.double(), offd, tau, mom, y, fl, y, grad_moments_in=gm)
    cell = torch.repeat_interleave(torch.arange(n_cells, device="cuda"), torch.from_numpy(counts).cuda())
    top = torch.zeros(n_cells, dtype=torch.float64, device="cuda")
    top.scatter_reduce_(0, cell, g64.abs().max(dim=0).values, "amax")
    err = (g32.double() - g64).abs().max(dim=0).values
    assert torch.isfinite(g32).all()
    assert (err <= 3e-5 * top[cell] + 1e-30).all()
