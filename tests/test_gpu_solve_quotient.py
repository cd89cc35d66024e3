"""eps2_hat / (tau theta) where tau theta is so small that its reciprocal overflows, the
quotient not: the solve scales as 1 / tau there too."""

import pytest

from test_gpu_solve_mixed import _moments

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("keep", [False, True])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [3, 3000])
def test_tiny_tau_theta(n, prec, keep):
    """theta about 2^-44, tau 2^-982: tau theta is a subnormal number good to 2^-48 or so
    (2^-1026), which eps2_hat's part of the coefficients (1e-3 of them) takes on."""
    from paper_2606_15622_gb300 import api
    m = _moments(n, n, scale=2.0**-22)
    p = api.default_params(pivot_rtol=1e-18)
    lu = torch.empty(api.lu_doubles(n), dtype=torch.float64, device="cuda") if keep else None
    y, f = [None] * 2, [None] * 2
    for i, k in enumerate((0, 982)):
        tau = torch.full((n,), 2.0**-k, dtype=torch.float64, device="cuda")
        y[i], f[i] = api.fp_closure_solve(m, tau, params=p, prec=prec, lu_out=lu)
    assert torch.equal(f[0], f[1])
    if prec == "fp64":
        assert (f[0] == 0).all()
    assert ((y[1] * 2.0**-982 - y[0]).norm(dim=1) <= 1e-13 * y[0].norm(dim=1)).all()
