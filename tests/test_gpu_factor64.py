"""FP64 block Thomas eliminated from both ends (factor64.cu) and its inward / outward substitutions at
the edges of their tilings: one, two and three columns (no chain, one chain, both), the row counts
where the kernel changes (16, 32, 256 and 512 padded rows) and panels that are not full."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# 1e-10 is the suite's bar for every FP64 path against the oracle
SHAPES = [(1, 1), (5, 2), (16, 3), (17, 1), (17, 4), (32, 9), (33, 2), (47, 3), (48, 1), (64, 10), (129, 5), (256, 3),
          (257, 6), (512, 4), (513, 3), (600, 2)]


@pytest.mark.parametrize("M,N", SHAPES)
@pytest.mark.parametrize("B", [1, 13])
def test_fp64_two_ended_factor(M, N, B):
    R = (1.0, 2.5, 2.5, 10.0)
    G, V = case(M, N, B, None, seed=M + N)
    ref = oracle.solve(M, N, G, *R, V, voltages=True)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    xb.set_option("orientation", "columns").set_option("algorithm", "thomas")
    I = torch.zeros((B, N), dtype=torch.float64, device="cuda")
    vW = torch.zeros((B, M, N), dtype=torch.float64, device="cuda")
    vB = torch.zeros_like(vW)
    for _ in range(2):  # a repeated factor reuses the counters and slots
        xb.factor("fp64")
        xb.solve(torch.from_numpy(V).cuda(), I, vWL=vW, vBL=vB)
        xb.sync()
        assert rel_err(I.cpu().numpy(), ref["I"]) <= 1e-10
        assert rel_err(vW.cpu().numpy(), ref["vWL"]) <= 1e-10
        assert rel_err(vB.cpu().numpy(), ref["vBL"]) <= 1e-10
    xb.destroy()
