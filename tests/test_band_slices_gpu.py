"""B^{-1} (Section 5.2) with a cluster of CTAs per subdomain where some planes are too narrow to
give every CTA rows.

Four subdomains whose planes are about ``narrow`` and ``wide`` rows wide: the split follows the
widest, so the narrow ones' clusters have CTAs without a 32-row block; at 192 rows the
assignment of six blocks to four CTAs leaves one out.  Oracle, tolerances and the
column's independence as in ``test_band_planes_gpu.py``.
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


@pytest.mark.parametrize("narrow,wide", [(1, 128), (32, 200), (40, 200), (70, 129), (96, 257), (192, 192)])
@pytest.mark.parametrize("split,threads", [(0, 0), (2, 512), (4, 256)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_bsolve_of_slices_without_rows(narrow, wide, split, threads, precision):
    nx, ny = narrow + wide + 2, 15
    P = slrgen.make_problem(f"slices-{narrow}-{wide}", (nx, ny), (2, 2), 0, kind="fv", coef_range=(0.5, 2.0))
    x, y = np.arange(nx * ny) % nx, np.arange(nx * ny) // nx
    P.part = (2 * (y >= ny // 2) + (x > narrow)).astype(np.int32)
    order = dd_order(P.rowptr, P.colind, P.part, P.nparts)
    f = np.random.default_rng(wide).standard_normal((order.n_I, 3))
    want = BSolver(split_blocks(P.rowptr, P.colind, P.val, order)[0], order.int_off).solve(f)
    g = SLR(P.rowptr, P.colind, P.val, P.part, P.nparts, k=0, precision=precision, nrhs_max=3, band_split=split,
            band_threads=threads)
    info = g.get_info()
    assert info["band_split"] == (split or (4 if wide <= 256 else 2)) and info["band_threads"] == (threads or 512)
    t = g.bsolve(torch.tensor(f, device="cuda")).cpu().numpy()
    tol = TOL64 if precision == "fp64" else tol32(info)
    assert np.abs(t - want).max() <= tol * np.abs(want).max()
    assert np.array_equal(g.bsolve(torch.tensor(f[:, 2], device="cuda")).cpu().numpy(), t[:, 2])
    g.close()
