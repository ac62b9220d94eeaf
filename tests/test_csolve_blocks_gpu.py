"""C solves of blocks of right-hand sides against single columns, at the widths where a kernel or
its accesses change."""
import numpy as np
import pytest
import torch

import slrgen
from paper_1505_04340_gb300 import SLR

pytestmark = pytest.mark.gpu


def cu(a):
    return torch.tensor(a, device="cuda")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nrhs", [8, 13, 16, 31, 64])
def test_csolve_block_widths_equal_single_columns(precision, nrhs):
    """Blocks whose rows do and do not start on 16-byte boundaries (8, 16, 64 against 13, 31), with one
    pass and several, and one large enough (64 columns of s = 24,696) to bring the solution to DD order
    in a pass of its own: every column equals the column solved alone, bit for bit."""
    P = slrgen.make_problem("m40", (40, 40, 40), (4, 4, 4), 4)
    g = SLR(P.rowptr, P.colind, P.val, P.part, P.nparts, k=0, precision=precision, nrhs_max=nrhs)
    gg = np.random.default_rng(nrhs).standard_normal((g.s, nrhs))
    y = g.csolve(cu(gg)).cpu().numpy()
    for c in {0, 7, nrhs // 2, nrhs - 1}:
        assert np.array_equal(g.csolve(cu(gg[:, c])).cpu().numpy(), y[:, c]), c
    g.close()
