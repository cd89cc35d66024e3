"""fp_step_host in FP64 with chunks of few cells: the bits of the unchunked calls, whatever the
number of chunks."""

import pytest
import torch

from paper_2606_15622_gb300 import populations as P
from paper_2606_15622_gb300 import surrogate as S
from test_gpu_pipeline import WEIGHTS, _pipeline, _reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells,n_chunks", [((80, 64), 4), ((80, 64), 16), ((20, 20), 3)])
def test_few_cells_a_chunk(cells, n_chunks):
    """Chunks below the count up to which a call gathers a cell by a whole warp, of calls above
    it (5,120 cells) and below it (400)."""
    pop = P.cavity(nx=cells[0], ny=cells[1])
    sur = S.Surrogate.load(WEIGHTS)
    vh = torch.from_numpy(pop.v64).pin_memory()
    ref = _reference(pop, vh.cuda(), "fp64", sur, 0.2, 5, 3)
    got = _pipeline(pop, vh, "fp64", sur, 0.2, 5, 3, n_chunks)
    for k in ref:
        assert torch.equal(got[k], ref[k].cpu()), k
