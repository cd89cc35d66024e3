"""The FP64 elimination where its rows are left out by the system's structure, its reciprocals
are at the ends of the exponent's range and its pivots sit in any row: the residual of the
solution against the oracle's matrix, with and without stored factors, and the adjoint by the
stored factors against the transposed elimination."""

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0**-53


def _moments(kind, n):
    from paper_2606_15622_gb300 import api
    rng = np.random.default_rng(n)
    off = torch.arange(0, 60 * n + 1, 60, dtype=torch.int64, device="cuda")
    v = rng.standard_normal((3, 60 * n)) * rng.permutation([1.0, 30.0, 0.02])[:, None]
    v += 0.2 * (v**2 - 1)
    m = api.fp_moments(torch.from_numpy(v).cuda(), off, prec="fp64").cpu().numpy()
    if kind == "diagonal":  # off-diagonal stresses exactly zero: zeros in every column
        m[:, [6, 7, 9]] = 0.0
    elif kind == "no third":
        m[:, 11:21] = 0.0
    elif kind == "no first":  # the first columns' own entries vanish: pivots from the rows below
        m[:, 5] = 0.0
    return m


@pytest.mark.parametrize("kind", ["plain", "diagonal", "no third", "no first"])
@pytest.mark.parametrize("n", [40, 1217, 3000])
def test_residual(kind, n):
    """Partial pivoting: |A y - r| <= 3 n rho u |A| |y| (n = 9, growth rho <= 10 on these) and
    a few roundings of the assembly."""
    from paper_2606_15622_gb300 import api
    m = _moments(kind, n)
    tau = np.random.default_rng(1).uniform(0.5, 2.0, n)
    tau[::7] = 1e-300
    tau[3::7] = 1e250
    md, td = torch.from_numpy(m).cuda(), torch.from_numpy(tau).cuda()
    lu = torch.empty(api.lu_doubles(n), dtype=torch.float64, device="cuda")
    y, f = api.fp_closure_solve(md, td, prec="fp64")
    y2, f2 = api.fp_closure_solve(md, td, prec="fp64", lu_out=lu)
    assert torch.equal(y, y2) and torch.equal(f, f2)
    ys, fs = y.cpu().numpy(), f.cpu().numpy()
    for c in np.nonzero(fs == 0)[0][::17]:
        A, r = O.assemble(m[c], tau[c])
        A, r = np.asarray(A).reshape(9, 9), np.asarray(r)
        size = np.abs(A).sum(1).max() * np.abs(ys[c]).max() + np.abs(r).max()
        assert np.abs(A @ ys[c] - r).max() <= 300 * U * size
    g = torch.randn(n, 9, dtype=torch.float64, device="cuda")
    v1, o1 = torch.zeros((3, 1), dtype=torch.float64, device="cuda"), torch.zeros_like(f, dtype=torch.int64)
    o1 = torch.cat([o1, o1[:1]])
    # without the cell's right-hand side the gradients hold lambda and Y alone
    a, _ = api.fp_closure_backward(v1, o1, td, md, y, f, g, want_grad_v=False)
    b, _ = api.fp_closure_backward(v1, o1, td, md, y, f, g, want_grad_v=False, lu=lu)
    a, b = a.cpu().numpy(), b.cpu().numpy()
    for c in np.nonzero(fs == 0)[0][::17]:
        kappa = np.linalg.cond(np.asarray(O.assemble(m[c], tau[c])[0]).reshape(9, 9))
        if kappa < 1e8:
            assert np.abs(a[c] - b[c]).max() <= 600 * U * kappa * np.abs(a[c]).max()


@pytest.mark.parametrize("tau", [5e-324, 1e-310, 1e-308, 3e-308, 1e-300, 2e307, 1e308, 1.7e308])
def test_tau_at_the_ends(tau):
    """tau's reciprocal overflows, is subnormal or is ordinary: a cell whose right-hand side is
    not finite is flagged, the others solve the oracle's system where tau theta is finite (a
    subnormal reciprocal is good to its last place)."""
    from paper_2606_15622_gb300 import api
    m = _moments("plain", 64)
    y, f = api.fp_closure_solve(torch.from_numpy(m).cuda(), torch.full((64,), tau, dtype=torch.float64, device="cuda"),
                                prec="fp64")
    y, f = y.cpu().numpy(), f.cpu().numpy()
    for c in range(0, 64, 9):
        with np.errstate(all="ignore"):
            A, r = O.assemble(m[c], tau)
            A, r = np.asarray(A).reshape(9, 9), np.asarray(r)
            if not np.isfinite(r).all():
                assert f[c] != 0
            elif f[c] == 0 and np.isfinite(tau * m[c, 4]):
                size = np.abs(A).sum(1).max() * np.abs(y[c]).max() + np.abs(r).max() + 1e-320
                assert np.abs(A / 1e3 @ y[c] - r / 1e3).max() <= 300 * U * size / 1e3 + 1e-318
