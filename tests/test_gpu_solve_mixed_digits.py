"""The mixed-precision solve's residual carries its digits: on well-conditioned cells the
refined coefficients agree with the FP64 solve far below FP32."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [200, 3000])
def test_well_conditioned_cells(n):
    """Skewed, anisotropic cells of 400 particles (condition of order 100).  One refinement
    leaves (2^-24 condition)^2 of the solution, about 4e-11, and the residual's own rounding
    (about 2^-44 of its terms) as much: 1e-9.  A residual good to FP32 only would leave
    2^-24 times the condition, 6e-6."""
    from paper_2606_15622_gb300 import api
    rng = np.random.default_rng(n)
    v = rng.standard_normal((3, 400 * n)) * np.array([[1.0], [1.3], [0.8]])
    v += 0.2 * (v**2 - 1)
    off = torch.arange(n + 1, device="cuda") * 400
    m = api.fp_moments(torch.from_numpy(v).cuda(), off, prec="fp64")
    tau = torch.linspace(0.5, 2.0, n, dtype=torch.float64, device="cuda")
    y64, f64 = api.fp_closure_solve(m, tau, prec="fp64")
    y32, f32 = api.fp_closure_solve(m, tau, prec="fp32")
    assert (f64 == 0).all() and (f32 == 0).all()
    assert not torch.equal(y64, y32)
    assert ((y32 - y64).norm(dim=1) / y64.norm(dim=1)).max() <= 1e-9
