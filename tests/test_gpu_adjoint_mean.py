"""The adjoint's FP32 particle pass does not lose digits to the cells' mean velocity."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_shifted_velocities():
    """Velocities on a grid of 2^-18, so that the shift by 16 is exact: c = v - U is the same
    number, and so is the error but for rounding luck (a quarter at most over 300,000
    particles).  U rounded to FP32 would add 2^-21 of c."""
    from paper_2606_15622_gb300 import api
    n_cells = 32768 + 100
    rng = np.random.default_rng(5)
    counts = np.array([(8, 12, 9, 7)[c % 4] for c in range(n_cells)])
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    n = int(off[-1])
    v0 = np.round(rng.standard_normal((3, n)) * 2**18) * 2.0**-18
    v0 = np.clip(v0, -4, 4)
    offd = torch.from_numpy(off).cuda()
    tau = torch.ones(n_cells, dtype=torch.float64, device="cuda")
    y = torch.zeros((n_cells, 9), dtype=torch.float64, device="cuda")
    fl = torch.full((n_cells,), api.FLAG_FEW, dtype=torch.int32, device="cuda")  # the closure's own part is zero
    gm = torch.from_numpy(rng.standard_normal((n_cells, 30))).cuda()
    err = []
    for shift in (0.0, 16.0):
        v = torch.from_numpy((v0 + shift).astype(np.float32)).cuda()
        assert np.array_equal(v.cpu().numpy().astype(np.float64), v0 + shift)
        mom = api.fp_moments(v.double(), offd, prec="fp64")
        _, g32 = api.fp_closure_backward(v, offd, tau, mom, y, fl, y, grad_moments_in=gm)
        _, g64 = api.fp_closure_backward(v.double(), offd, tau, mom, y, fl, y, grad_moments_in=gm)
        err.append(float((g32.double() - g64).norm() / g64.norm()))
    assert err[1] <= 1.25 * err[0]
