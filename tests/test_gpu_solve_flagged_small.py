"""Small FP64 solves (a half warp a cell) of flagged cells: no elimination for a warp whose
cells are all flagged, and the same results for flagged cells beside others."""

import pytest

from test_gpu_gather_fp64_tasks import _seconds
from test_gpu_solve_mixed import _moments

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_flagged_cells_are_not_solved():
    """Loading 400 cells and writing the linear drift is well under two thirds of the
    elimination's chain (12 us)."""
    from paper_2606_15622_gb300 import api
    m = _moments(400, 2)
    tau = torch.full((400,), 0.5, dtype=torch.float64, device="cuda")
    y, f = torch.empty(400, 9, dtype=torch.float64, device="cuda"), torch.empty(400, dtype=torch.int32, device="cuda")
    t = []
    for few in (5, 10**6):
        p = api.default_params(min_particles=few)
        t.append(_seconds(lambda: api.fp_closure_solve(m, tau, params=p, prec="fp64", coeffs_out=y, flags_out=f)))
        assert (f == (api.FLAG_FEW if few > 5 else 0)).all()
    assert t[1] <= 0.65 * t[0]


@pytest.mark.parametrize("n", [1, 2, 7, 400])
@pytest.mark.parametrize("every", [1, 2, 3])
def test_flagged_beside_others(n, every):
    """Cell c has the same results alone as among others."""
    from paper_2606_15622_gb300 import api
    m = _moments(n, 4)
    m[::every, 0] = 2
    tau = torch.linspace(0.5, 2.0, n, dtype=torch.float64, device="cuda")
    y, f = api.fp_closure_solve(m, tau, prec="fp64")
    assert (f[::every] == api.FLAG_FEW).all()
    want = torch.zeros(n, 9, dtype=torch.float64, device="cuda")
    want[:, [0, 3, 5]] = -1.0 / tau[:, None]
    assert torch.equal(y[::every], want[::every])
    for c in range(0, n, max(1, n // 7)):
        y1, f1 = api.fp_closure_solve(m[c:c + 1], tau[c:c + 1], prec="fp64")
        assert torch.equal(y1, y[c:c + 1]) and torch.equal(f1, f[c:c + 1])
