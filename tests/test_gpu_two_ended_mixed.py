"""The FP32 factor and substitutions with two elimination chains at the edges of their tilings: one to
four columns (no chain, one chain, both), blocks of one and of two 128-row halves, panels that are not
full, each factor kernel (cluster: two chains, group: one) with each substitution kernel."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 1e-8 is the suite's bar for refined currents; node voltages follow the same certificate
@pytest.mark.parametrize("M,N", [(33, 1), (40, 2), (100, 3), (128, 4), (129, 2), (256, 3)])
@pytest.mark.parametrize("factor", [0, 1])
@pytest.mark.parametrize("sweep", [0, 1])
def test_mixed_two_ended(M, N, factor, sweep):
    R = (1.0, 2.5, 2.5, 10.0)
    B = 65
    G, V = case(M, N, B, None, seed=M + N)
    ref = oracle.solve(M, N, G, *R, V, voltages=True)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    xb.set_option("orientation", "columns").set_option("algorithm", "thomas")
    xb.set_option("factor_kernel", factor).set_option("sweep_kernel", sweep)
    I = torch.zeros((B, N), dtype=torch.float64, device="cuda")
    vW = torch.zeros((B, M, N), dtype=torch.float64, device="cuda")
    vB = torch.zeros_like(vW)
    for b in (B, 1):
        xb.factor("fp32_ir")
        xb.solve(torch.from_numpy(V[:b]).cuda(), I[:b], vWL=vW[:b], vBL=vB[:b], tol=1e-9)
        assert rel_err(I[:b].cpu().numpy(), ref["I"][:b]) <= 1e-8
        assert rel_err(vW[:b].cpu().numpy(), ref["vWL"][:b]) <= 1e-8
        assert rel_err(vB[:b].cpu().numpy(), ref["vBL"][:b]) <= 1e-8
    xb.destroy()
