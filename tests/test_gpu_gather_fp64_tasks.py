"""The FP64 gather's warps take whole tasks of four cells: a few more cells a warp cost a few
more cells' time."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _seconds(call, reps=20):
    """Device time of a call, the best of three rounds of `reps` in one graph."""
    for _ in range(3):
        call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(reps):
            call()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(3):
        graph.replay()
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / reps)
    return best


def test_nine_cells_a_warp_beside_eight():
    """FP64 sums (a cold beam: bound by the FP64 pipe, so by the number of tasks).  Nine
    cells a warp are 12.5 % more work than eight; three tasks instead of two are 50 %."""
    from paper_2606_15622_gb300 import api
    warps = 12 * torch.cuda.get_device_properties(0).multi_processor_count
    t = []
    for per_warp in (8, 9):
        n = per_warp * warps
        off = torch.arange(n + 1, device="cuda") * 48
        v = torch.randn(3, n * 48, dtype=torch.float64, device="cuda")
        v[1] += 1e3
        m = torch.empty(n, 30, dtype=torch.float64, device="cuda")
        t.append(_seconds(lambda: api.fp_moments(v, off, prec="fp64", moments_out=m)))
    assert t[1] <= 1.3 * t[0]
