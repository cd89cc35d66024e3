"""The FP64 gather on cells with heavy tails (outliers, hot tails) beside Maxwellian ones:
every sum within its bound."""

import numpy as np
import pytest

from test_fixed_point_lanes_host import HEAVY, PAIRS, TRIPLES, bounds, heavy

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells", [100, 2500])
@pytest.mark.parametrize("kind", HEAVY, ids=str)
def test_heavy_tails(kind, n_cells):
    """Reference in long double about the call's own means."""
    from paper_2606_15622_gb300 import api
    rng = np.random.default_rng(n_cells)
    cells = [heavy(kind, (9, 16, 30, 100, 300, 1000)[c % 6] if c < 60 else 30, rng) if c % 4 else
             rng.standard_normal((3, 40)) for c in range(n_cells)]
    off = np.concatenate([[0], np.cumsum([x.shape[1] for x in cells])]).astype(np.int64)
    m6 = torch.empty(n_cells, dtype=torch.float64, device="cuda")
    v = torch.from_numpy(np.concatenate(cells, axis=1)).cuda()
    m = api.fp_moments(v, torch.from_numpy(off).cuda(), prec="fp64", m6_out=m6).cpu().numpy()
    got = np.concatenate([m[:, 5:], m6.cpu().numpy()[:, None]], axis=1)
    for k, x in enumerate(cells[:120]):
        c = x.astype(np.longdouble) - m[k, 1:4].astype(np.longdouble)[:, None]
        r2 = (c * c).sum(0)
        t = np.array([c[i] * c[j] for i, j in PAIRS] + [c[i] * c[j] * c[l] for i, j, l in TRIPLES]
                     + [r2 * c[i] * c[j] for i, j in PAIRS] + [r2 * r2 * c[i] for i in range(3)] + [r2 * r2 * r2])
        n = x.shape[1]
        off_by = np.abs(got[k] * n - t.sum(1))
        assert (off_by <= bounds(np.abs(t).sum(1), np.abs(c).max(1), n)).all(), k
