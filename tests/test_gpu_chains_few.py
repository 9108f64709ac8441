"""Refinement and node voltages with the bit-line chains cut into row segments (few vectors): one row to
1000, more segments than rows, ragged segments and batches, both formulations (sources on the word lines
and, blocked over rows, on the bit lines)."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = (1.0, 2.5, 2.5, 10.0)


# the suite's bars: 1e-8 for refined results, 1e-10 for FP64
@pytest.mark.parametrize("precision,bar", [("fp32_ir", 1e-8), ("fp64", 1e-10)])
@pytest.mark.parametrize("orientation", ["columns", "rows"])
@pytest.mark.parametrize("M,N", [(1, 3), (7, 2), (33, 1), (100, 5), (257, 3), (1000, 2)])
def test_chains_few(M, N, orientation, precision, bar):
    G, V = case(M, N, 40, None, seed=M + 2 * N)
    ref = oracle.solve(M, N, G, *R, V, voltages=True)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    xb.set_option("orientation", orientation)
    xb.factor(precision)
    for b in (1, 3, 40):
        I = torch.zeros((b, N), dtype=torch.float64, device="cuda")
        vW = torch.zeros((b, M, N), dtype=torch.float64, device="cuda")
        vB = torch.zeros_like(vW)
        xb.solve(torch.from_numpy(V[:b].copy()).cuda(), I, vWL=vW, vBL=vB, tol=1e-9)
        xb.sync()
        assert rel_err(I.cpu().numpy(), ref["I"][:b]) <= bar
        assert rel_err(vW.cpu().numpy(), ref["vWL"][:b]) <= bar
        assert rel_err(vB.cpu().numpy(), ref["vBL"][:b]) <= bar
    xb.destroy()
