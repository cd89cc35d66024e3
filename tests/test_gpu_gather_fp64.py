"""The FP64 gather against the oracle where its forms meet: cell sizes around the FP64
few-particle limit, the lanes' rounds and the fixed-point block, warp-per-cell and
eight-lane launches, velocities of both types, and cells that mix the fixed-point and
the FP64 form in one warp task."""

import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _population(counts, scale, seed):
    rng = np.random.default_rng(seed)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    v = rng.standard_normal((3, int(off[-1]))) * np.asarray(scale)[:, None] + np.array([3.0, -1.0, 0.0])[:, None]
    return v, off


def _check(v, off, tol):
    """Every moment within tol of <|c|^k> of its order (the cell means within tol of the
    largest speed)."""
    from paper_2606_15622_gb300 import api
    n = off.size - 1
    m6 = torch.empty(n, dtype=torch.float64, device="cuda")
    got = api.fp_moments(torch.from_numpy(v).cuda(), torch.from_numpy(off).cuda(), prec="fp64", m6_out=m6)
    got, m6 = got.cpu().numpy(), m6.cpu().numpy()
    v = v.astype(np.float64)
    ref = O.moments(v, off)
    np.testing.assert_array_equal(got[:, 0], ref[:, 0])
    for c in range(n):
        x = v[:, off[c]:off[c + 1]]
        if x.shape[1] == 0:
            assert (got[c, 1:] == 0).all() and m6[c] == 0
            continue
        if not np.isfinite(x).all():
            assert not np.isfinite(got[c, 4])
            continue
        r = np.linalg.norm(x - x.mean(axis=1, keepdims=True), axis=0)
        slot = np.concatenate([np.full(3, np.abs(x).max()), np.full(7, (r**2).mean()), np.full(10, (r**3).mean()),
                               np.full(6, (r**4).mean()), np.full(3, (r**5).mean())])
        # a mean off by an ulp of the speed moves a moment by that over the spread
        cond = 1 + np.abs(x).max() / max(r.max(), 1e-300)
        assert (np.abs(got[c, 1:] - ref[c, 1:]) <= tol * cond * slot + 1e-300).all(), c
        assert abs(m6[c] - (r**6).mean()) <= 10 * tol * cond * (r**6).mean() + 1e-300, c


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("n_cells", [1, 5, 3001])
def test_sizes(dtype, n_cells):
    """1e-14: some ten FP64 roundings of each side in moments of its order."""
    sizes = [0, 1, 2, 4, 7, 8, 9, 15, 16, 17, 31, 33, 64, 119, 120, 121, 240, 241, 257, 1000]
    counts = [sizes[(7 * c + n_cells) % len(sizes)] for c in range(n_cells)]
    v, off = _population(counts, (1.0, 1.7, 0.6), n_cells)
    _check(v.astype(dtype), off, 1e-14)


@pytest.mark.parametrize("n_cells", [64, 4000])
def test_forms_mixed_in_a_task(n_cells):
    """Neighbouring cells of plain, thin, cold, constant, tiny, huge and non-finite
    velocities: each takes its own form."""
    counts = [20 + 3 * (c % 9) for c in range(n_cells)]
    v, off = _population(counts, (1.0, 1.0, 1.0), 11)
    for c in range(n_cells):
        x = v[:, off[c]:off[c + 1]]
        k = c % 8
        if k == 1:
            x[2] *= 1e-3
        elif k == 2:
            x[0] += 1e4
        elif k == 3:
            x[1] = 0.25
        elif k == 4:
            x *= 1e-45
        elif k == 5:
            x *= 1e41
        elif k == 6 and c % 16 == 6:
            x[1, 3] = np.nan if c % 32 == 6 else np.inf
    _check(v, off, 1e-14)
