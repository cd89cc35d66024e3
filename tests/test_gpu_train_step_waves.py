"""The training step over the waves of its backward pass (a tile of 128 rows an SM)."""

import pytest

from test_gpu_gather_fp64_tasks import _seconds

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _step(rows):
    from paper_2606_15622_gb300 import surrogate
    s = surrogate.Surrogate()
    s.init_params(0)
    tr = surrogate.Trainer(s, batch=rows)
    g = torch.Generator(device="cuda").manual_seed(rows)
    x = torch.randn(rows, 32, generator=g, device="cuda").bfloat16()
    t = torch.randn(rows, 9, generator=g, device="cuda")
    aux = torch.rand(rows, 16, generator=g, device="cuda")
    return lambda: tr.step(x, t, aux, 1.0 / rows)


def test_full_waves():
    """Two full waves beside one and a third: half as many rows again, the same number of
    waves and a third more partial sums to add, so a third longer at most."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    partial, full = _seconds(_step(128 * (sms + sms // 3))), _seconds(_step(128 * 2 * sms))
    assert full <= 1.4 * partial
