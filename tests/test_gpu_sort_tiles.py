"""The cell sort at the edges of its tiles, histogram blocks and scan parts, with keys that
take either ranking (few runs in a warp, many distinct digits), an input that is not
16-byte aligned, and velocities of both types."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 4095, 4096, 4097, 16383, 16385, 512 * 4096 - 3, 513 * 4096 + 7, 4 * 512 * 4096 + 1])
@pytest.mark.parametrize("order", ["sorted", "random", "constant", "comb", "outside"])
@pytest.mark.parametrize("n_cells", [1, 300, 70001])
def test_sort(n, order, n_cells):
    from paper_2606_15622_gb300 import api
    g = torch.Generator(device="cuda").manual_seed(n + n_cells)
    i = torch.arange(n, device="cuda")
    key = {"sorted": lambda: i * n_cells // n, "constant": lambda: torch.full_like(i, n_cells // 2),
           "comb": lambda: i * 7919 % n_cells,
           "random": lambda: torch.randint(0, n_cells, (n,), generator=g, device="cuda"),
           "outside": lambda: torch.randint(-2, n_cells + 3, (n,), generator=g, device="cuda")}[order]()
    at = n % 4  # elements from a 16-byte boundary
    cell = torch.empty(n + 4, dtype=torch.int32, device="cuda")[at:at + n].copy_(key)
    v = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float32 if n % 2 else torch.float64)
    perm, off, vs = api.fp_sort_by_cell(cell, n_cells, v=v)
    k = torch.where((key >= 0) & (key < n_cells), key, torch.full_like(key, n_cells))
    ks, want = torch.sort(k, stable=True)
    assert torch.equal(perm.long(), want)
    assert torch.equal(off, torch.searchsorted(ks, torch.arange(n_cells + 1, device="cuda")))
    assert torch.equal(vs, v[:, want])
