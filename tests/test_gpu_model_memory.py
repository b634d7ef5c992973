"""GPU: a model whose cell records fill whole 2 MiB pages takes no page beyond them.  What is
kept beside the records is small and shares the page of the other small allocations; in one
allocation with them it cost a page, and a creation 10 % longer."""
import gc

import pytest

from paper_2512_01283_gb300 import build as B
from paper_2512_01283_gb300 import mcrt as M
from paper_2512_01283_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 128])
def test_cells_of_whole_pages_take_no_page_more(n):
    import torch

    B.build()
    host = W.dichroic_slab(n=n)
    model = dict(host, **{k: torch.from_numpy(host[k]).cuda() for k in ("kappa_abs", "kappa_sca", "bfield")
                          if host.get(k) is not None})
    first = M.Model(model)  # loads the set-up kernels and opens the page of the small allocations
    gc.collect()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    second = M.Model(model)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    second.close()
    first.close()
    assert 32 * n ** 3 <= taken < 32 * n ** 3 + (2 << 20)
