"""FP64 factors by the group kernel (factor.cu), which takes over on devices with too few SMs for
factor64.cu: one block (up to 32 rows), groups of two-row blocks, blocks with several rows."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 1e-10 is the suite's bar for every FP64 path against the oracle
@pytest.mark.parametrize("M,N", [(1, 1), (16, 3), (17, 4), (32, 9), (33, 2), (64, 10), (257, 3), (600, 2)])
def test_group_factor(M, N, monkeypatch):
    monkeypatch.setenv("XBAR_FACTOR", "group")
    R = (1.0, 2.5, 2.5, 10.0)
    G, V = case(M, N, 13, None, seed=M + N)
    ref = oracle.solve(M, N, G, *R, V, voltages=True)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    xb.set_option("orientation", "columns").set_option("algorithm", "thomas")
    for B in (13, 1):
        I = torch.zeros((B, N), dtype=torch.float64, device="cuda")
        vB = torch.zeros((B, M, N), dtype=torch.float64, device="cuda")
        xb.factor("fp64")
        xb.solve(torch.from_numpy(np.ascontiguousarray(V[:B])).cuda(), I, vBL=vB)
        xb.sync()
        assert rel_err(I.cpu().numpy(), ref["I"][:B]) <= 1e-10
        assert rel_err(vB.cpu().numpy(), ref["vBL"][:B]) <= 1e-10
    monkeypatch.delenv("XBAR_FACTOR")
    xb.factor("fp64").solve(torch.from_numpy(np.ascontiguousarray(V[:1])).cuda(), I)  # and back
    xb.sync()
    assert rel_err(I.cpu().numpy(), ref["I"][:1]) <= 1e-10
    xb.destroy()
