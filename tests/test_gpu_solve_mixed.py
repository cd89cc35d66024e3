"""The mixed-precision solve (FP32 factors, residual in pairs of FP32) against the FP64 solve
of the same moments: cells of the three flows' kinds, warps with one, a few and many cells
that go back to the FP64 elimination, moments and tau at the ends of the pairs' range and
beyond it, and calls small enough for the half-warp FP64 kernel."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _moments(n, seed, scale=1.0, few_every=0):
    from paper_2606_15622_gb300 import api
    rng = np.random.default_rng(seed)
    counts = np.full(n, 60)
    if few_every:
        counts[::few_every] = 9  # ill-conditioned cells
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    v = rng.standard_normal((3, int(off[-1]))) * np.array([[1.0], [1.3], [0.8]])
    v += 0.2 * (v**2 - 1)
    return api.fp_moments(torch.from_numpy(v * scale).cuda(), torch.from_numpy(off).cuda(), prec="fp64")


@pytest.mark.parametrize("n", [1, 31, 33, 1216, 1217, 5000])
@pytest.mark.parametrize("few_every", [0, 2, 13, 40])
def test_against_fp64(n, few_every):
    """1e-7 of a cell's coefficients: a correction of at most 1e-4 of them whose own solve
    is good to 2^-24 times a condition of order 1e3; cells eliminated in FP64 are equal."""
    from paper_2606_15622_gb300 import api
    m = _moments(n, n, few_every=few_every)
    tau = torch.linspace(0.5, 2.0, n, dtype=torch.float64, device="cuda")
    # FP32 mode's pivot floor in the FP64 mode: the same singularity threshold
    y64, f64 = api.fp_closure_solve(m, tau, params=api.default_params(pivot_rtol=1e-6), prec="fp64")
    y32, f32 = api.fp_closure_solve(m, tau, prec="fp32")
    assert torch.equal(f64, f32)
    err = (y32 - y64).norm(dim=1) / y64.norm(dim=1)
    assert err.max() <= 1e-7


@pytest.mark.parametrize("scale", [2.0**-9, 2.0**9, 2.0**-12, 2.0**12, 1e-20, 1e9])
def test_scaled_units(scale):
    """Velocities in other units, within and beyond the pairs' range (theta of 2^+-20)."""
    from paper_2606_15622_gb300 import api
    m = _moments(200, 3, scale=scale)
    tau = torch.full((200,), 0.7, dtype=torch.float64, device="cuda")
    p = api.default_params(pivot_rtol=1e-6)
    y64, f64 = api.fp_closure_solve(m, tau, params=p, prec="fp64")
    y32, f32 = api.fp_closure_solve(m, tau, prec="fp32")
    assert torch.equal(f64, f32)
    err = (y32 - y64).norm(dim=1) / y64.norm(dim=1).clamp(min=1e-300)
    assert err.max() <= 1e-7


def test_flagged_cells_take_the_linear_drift():
    from paper_2606_15622_gb300 import api
    m = _moments(70, 5)
    m[3, 0], m[10, 4], m[20, 12], m[40, 0] = 3, -1.0, float("nan"), 4
    tau = torch.full((70,), 2.0, dtype=torch.float64, device="cuda")
    tau[50] = float("inf")
    y, f = api.fp_closure_solve(m, tau, prec="fp32")
    want = torch.zeros(9, dtype=torch.float64, device="cuda")
    want[[0, 3, 5]] = -0.5
    for c, flag in ((3, api.FLAG_FEW), (10, api.FLAG_SINGULAR), (20, api.FLAG_NONFINITE), (40, api.FLAG_SINGULAR)):
        assert int(f[c]) == flag and torch.equal(y[c], want)
    assert int(f[50]) == api.FLAG_NONFINITE and (y[50] == 0).all()
    assert (f == 0).sum() == 65
