"""The mixed-precision solve over the whole range of tau: the coefficients scale as 1 / tau."""

import pytest

from test_gpu_solve_mixed import _moments

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 5000])
@pytest.mark.parametrize("k", [-600, -120, -24, -21, -19, 19, 21, 24, 120, 600])
def test_power_of_two_of_tau(n, k):
    """tau enters the right-hand side only, as 1 / tau: tau 2^k gives the same bits, their
    exponents less k."""
    from paper_2606_15622_gb300 import api
    m = _moments(n, n, few_every=13)
    tau = torch.linspace(0.3, 3.0, n, dtype=torch.float64, device="cuda")
    y0, f0 = api.fp_closure_solve(m, tau, prec="fp32")
    y, f = api.fp_closure_solve(m, tau * 2.0**k, prec="fp32")
    assert torch.equal(f, f0)
    assert torch.equal(y * 2.0**k, y0)


def test_the_ends_of_tau():
    """Where 2^-k y leaves the double range: as the FP64 solve decides."""
    from paper_2606_15622_gb300 import api
    m = _moments(64, 1)
    tau = torch.tensor([5e-324, 1e-310, 1e-300, 1e300], dtype=torch.float64, device="cuda").repeat(16)
    y64, f64 = api.fp_closure_solve(m, tau, params=api.default_params(pivot_rtol=1e-6), prec="fp64")
    y32, f32 = api.fp_closure_solve(m, tau, prec="fp32")
    assert torch.equal(f32, f64)
    assert torch.equal(y32, y64)
