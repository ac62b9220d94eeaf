"""Calls whose kernels start before the stores of the ones ahead are flushed, against the same calls with plain edges.

Outside stream capture the kernels of a call are dependent launches; a captured call has plain
edges.  Calls back to back, each on what the
one before has just written, give bit for bit what the captured call gives on the same input.
"""
import numpy as np
import pytest

import slrgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1505_04340_gb300 import SLR  # noqa: E402

TF32 = dict(u_dtype="tf32", band_mma="tf32")
BF16 = dict(u_dtype="bf16", band_mma="bf16")


@pytest.mark.parametrize("precision,nrhs,options", [
    ("fp64", 1, {}), ("fp64", 3, {}), ("fp64", 8, {}), ("fp64", 2, dict(zform=True)), ("fp64", 1, dict(c_persistent=True)),
    ("mixed", 1, {}), ("mixed", 2, {}), ("mixed", 5, {}), ("mixed", 16, {}), ("mixed", 3, dict(c_top_zone=False)),
    ("mixed", 1, dict(zform=True)), ("mixed", 9, dict(zform=True)), ("mixed", 1, dict(c_persistent=True)),
    ("mixed", 3, dict(c_persistent=True, c_top_zone=False)),
    ("mixed", 8, TF32), ("mixed", 16, TF32), ("mixed", 33, TF32), ("mixed", 64, TF32), ("mixed", 16, BF16)])
def test_calls_in_a_row_equal_plain_edges(precision, nrhs, options):
    P = slrgen.make_problem("m24", (24, 24, 24), (2, 2, 2), 4)
    g = SLR(P.rowptr, P.colind, P.val, P.part, P.nparts, k=8, lanczos_steps=12, precision=precision, nrhs_max=nrhs,
            **options)
    side = torch.cuda.Stream()
    for f, rows in ((g.apply, P.n), (g.bsolve, g.n_interior), (g.csolve, g.s), (g.stilde_solve, g.s)):
        x = torch.tensor(np.random.default_rng(nrhs).standard_normal((nrhs, rows)), device="cuda").t()
        if nrhs == 1:
            x = x[:, 0].contiguous()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            held = x.clone(memory_format=torch.preserve_format)
            ins, outs = [], []
            for _ in range(6):
                y = f(x)
                ins.append(x)
                outs.append(y)
                x = 0.5 * x + y
            side.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                z = f(held)
            for x, y in zip(ins, outs):
                held.copy_(x)
                graph.replay()
                side.synchronize()
                assert torch.equal(z, y), f.__name__
    g.close()
