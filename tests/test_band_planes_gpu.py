"""B^{-1} (Section 5.2) at the plane widths where the band kernels' tiles end.

Each case has four subdomains whose planes are W and W + 1 rows wide: around the
32-row blocks, the groups of 16 columns (W <= 64: four warps per subdomain) and of 8
columns, the first width of the wider kernel, and single columns.  "skew" cuts the
subdomains along a ragged line, so that the last plane of a subdomain is not full.
The oracle's banded Cholesky is the reference; FP64 to 1e-10 (the inverted blocks'
rounding is bounded by kappa(D_J) eps, 1e-13 here), FP32 to the bound of
``tests/tolerances.py``; a column solved alone equals its column of a block bit for bit.
"""
import numpy as np
import pytest

import slrgen
from oracle.slr_oracle import BSolver, dd_order, split_blocks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1505_04340_gb300 import SLR  # noqa: E402

from tolerances import TOL64, tol32  # noqa: E402


def problem(W, c, skew):
    P = slrgen.make_problem(f"planes-{W}x{c}", (2 * W + 3, 2 * c + 3), (2, 2), 0, kind="fv", coef_range=(1e-2, 1e2))
    if skew:
        nx, ny = P.dims
        x, y = np.arange(nx * ny) % nx, np.arange(nx * ny) // nx
        P.part = (2 * (y >= ny // 2 + (x // 3) % 2) + (x >= nx // 2 + y % 3)).astype(np.int32)
    return P


@pytest.mark.parametrize("W,c,skew", [
    (1, 4, False), (3, 1, False), (4, 6, True), (7, 3, False), (15, 15, False), (16, 2, True), (31, 5, False),
    (32, 4, True), (47, 3, False), (48, 9, True), (63, 8, False), (62, 7, True)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_bsolve_at_tile_edges(W, c, skew, precision):
    P = problem(W, c, skew)
    order = dd_order(P.rowptr, P.colind, P.part, P.nparts)
    f = np.random.default_rng(W).standard_normal((order.n_I, 11))
    want = BSolver(split_blocks(P.rowptr, P.colind, P.val, order)[0], order.int_off).solve(f)
    g = SLR(P.rowptr, P.colind, P.val, P.part, P.nparts, k=0, precision=precision, nrhs_max=11)
    tol = TOL64 if precision == "fp64" else tol32(g.get_info())
    for r in (11, 7, 6, 5, 3, 2, 1):       # launches of 8 + 3 columns, and each narrower width
        t = g.bsolve(torch.tensor(f[:, :r], device="cuda")).cpu().numpy()
        assert np.abs(t - want[:, :r]).max() <= tol * np.abs(want[:, :r]).max(), r
        if r == 11:
            block = t
        assert np.array_equal(t, block[:, :r]), r
    g.close()


@pytest.mark.parametrize("W,c", [(65, 4), (96, 3), (128, 2), (224, 1), (225, 4), (255, 3), (257, 3)])
@pytest.mark.parametrize("split,threads", [(1, 512), (1, 256), (2, 256), (4, 256), (4, 512)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_bsolve_of_wide_planes(W, c, split, threads, precision):
    """The wider kernel at its first width and around whole row blocks, for each split and CTA size (a
    slice holds at most 256 rows: the last width needs two)."""
    if W > 256 and split == 1:
        split = 2
    P = problem(W, c, False)
    order = dd_order(P.rowptr, P.colind, P.part, P.nparts)
    f = np.random.default_rng(W).standard_normal((order.n_I, 11))
    want = BSolver(split_blocks(P.rowptr, P.colind, P.val, order)[0], order.int_off).solve(f)
    g = SLR(P.rowptr, P.colind, P.val, P.part, P.nparts, k=0, precision=precision, nrhs_max=11, band_split=split,
            band_threads=threads)
    info = g.get_info()
    assert (info["band_split"], info["band_threads"]) == (split, threads)
    tol = TOL64 if precision == "fp64" else tol32(info)
    for r in (11, 7, 6, 5, 3, 2, 1):
        t = g.bsolve(torch.tensor(f[:, :r], device="cuda")).cpu().numpy()
        assert np.abs(t - want[:, :r]).max() <= tol * np.abs(want[:, :r]).max(), r
        if r == 11:
            block = t
        assert np.array_equal(t, block[:, :r]), r
    g.close()
