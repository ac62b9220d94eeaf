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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nrhs", [1, 8])
@pytest.mark.parametrize("side", [False, True])
def test_applies_in_a_row_equal_applies_alone(precision, nrhs, side):
    """An apply's kernels start before the ones ahead of them have ended: calls back to back, each on
    an input that a kernel on the same stream has just written and into buffers that the call
    before still uses, give bit for bit what they give one at a time."""
    P = slrgen.make_problem("m24", (24, 24, 24), (2, 2, 2), 4)
    g = SLR(P.rowptr, P.colind, P.val, P.part, P.nparts, k=4, lanczos_steps=6, precision=precision, nrhs_max=nrhs)
    r = cu(np.random.default_rng(3).standard_normal((nrhs, P.n))).t()
    r = r[:, 0].contiguous() if nrhs == 1 else r
    with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.default_stream()):
        torch.cuda.synchronize()
        row, x = [], r
        for _ in range(8):
            x = x + g.apply(x)
            row.append(x)
        torch.cuda.synchronize()
        x = r
        for y in row:
            z = g.apply(x)
            torch.cuda.synchronize()
            x = x + z
            torch.cuda.synchronize()
            assert torch.equal(x, y)
    g.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nrhs", [2, 3, 5, 6, 7, 11])
def test_csolve_last_pass_widths_equal_single_columns(precision, nrhs):
    """Widths whose last pass over the top levels' inverse is narrower than the ones before: every column
    equals the column solved alone, bit for bit."""
    P = slrgen.make_problem("m32", (32, 32, 32), (2, 2, 2), 4)
    g = SLR(P.rowptr, P.colind, P.val, P.part, P.nparts, k=0, precision=precision, nrhs_max=nrhs)
    assert g.get_info()["c_top_positions"] > 0
    gg = np.random.default_rng(nrhs).standard_normal((g.s, nrhs))
    y = g.csolve(cu(gg)).cpu().numpy()
    for c in range(nrhs):
        assert np.array_equal(g.csolve(cu(gg[:, c])).cpu().numpy(), y[:, c]), c
    g.close()
