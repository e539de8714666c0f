"""The d-choices kernel at the edges of its groups of four balls, its tiles of
choices and its trials per CTA, against the oracle."""

import numpy as np
import pytest

from oracle import oracle as O
from parity_harness import lib_ready

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    lib_ready()


@pytest.mark.parametrize("n,m,d,trials", [(3, 3, 1, 1), (2, 257, 1, 151), (5, 127, 2, 152), (2, 129, 2, 153),
                                          (1, 6, 3, 40), (9, 85, 3, 2000), (256, 254, 4, 4864), (33, 65, 4, 4865),
                                          (17, 97, 5, 305), (40, 43, 63, 10)])
def test_potc_tile_edges(n, m, d, trials):
    import torch
    from paper_2602_06502_gb300 import dualmap as D
    out = torch.zeros(trials, dtype=torch.int32, device="cuda")
    assert D.dm_potc_max_loads(n, m, d, trials, 77 + m, out) == 0
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().astype(np.uint32), O.potc_max_loads(n, m, d, trials, 77 + m))
