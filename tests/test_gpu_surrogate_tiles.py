"""The learned closures' later tiles (inputs formed by the forming warps beside the network)
against the same cells in calls of one tile a group (inputs formed before the first layer):
bit for bit, with unusual values anywhere in the rows."""

import os

import numpy as np
import pytest
import torch

from paper_2606_15622_gb300 import api, surrogate as S

pytestmark = pytest.mark.gpu

W = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_15622_gb300", "weights")
BAD = [np.nan, np.inf, -np.inf, 0.0, -0.0, -1.0, 1e39, -1e39, 3e38, 1e-40, 5e-324, 1e300]


def _rows(n, lite):
    rng = np.random.default_rng(n)
    counts = rng.integers(15, 40, 300)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    v = torch.from_numpy(rng.standard_normal((3, int(off[-1])))).cuda()
    off = torch.from_numpy(off).cuda()
    m = (api.fp_moments_lite(v.float(), off) if lite else api.fp_moments(v, off, prec="fp64")).cpu().numpy()
    m = m[np.arange(n) % 300]
    m[:, 5:] *= 1 + 0.01 * rng.standard_normal((n, m.shape[1] - 5))  # every row its own
    tau = rng.uniform(0.5, 2.0, n)
    for r in range(3, n, 11):
        m[r, rng.integers(m.shape[1])] = BAD[rng.integers(len(BAD))]
    for r in range(7, n, 101):
        tau[r] = BAD[rng.integers(len(BAD))]
    return torch.from_numpy(m).cuda(), torch.from_numpy(tau).cuda()


@pytest.mark.parametrize("extra", [1, 128, 129, 257])
@pytest.mark.parametrize("turns", [1, 2, 3])
@pytest.mark.parametrize("lite", [False, True])
def test_later_tiles_equal_first_tiles(lite, turns, extra):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = turns * sms * 256 + extra
    m, tau = _rows(n, lite)
    s = S.Surrogate.load(os.path.join(W, "surrogate_lite.fpw" if lite else "surrogate_full.fpw"))
    run = s.closure_lite if lite else s.closure
    y, fl = run(m, tau)
    step = sms * 256  # one tile a group
    parts = [run(m[i:i + step].contiguous(), tau[i:i + step].contiguous()) for i in range(0, n, step)]
    y1, fl1 = torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])
    assert torch.equal(fl, fl1)
    assert torch.equal(y.view(torch.int64), y1.view(torch.int64))
    x, f0 = (s.lite_features if lite else s.features)(m, tau)
    assert torch.equal(fl & api.FLAG_RANGE, f0 & api.FLAG_RANGE)
