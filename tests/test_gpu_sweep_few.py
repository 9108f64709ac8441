"""Substitutions of a few vectors on clusters (sweep_few.cu): every panel width and rows-per-block choice,
one to five columns (no chain, one, both; the columns around the meeting one), ragged rows and batches,
currents alone and with node voltages, and the entry point without allocation."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = (1.0, 2.5, 2.5, 10.0)
BATCHES = [1, 2, 3, 8, 13, 33, 64]
# (M, N): 1 to 16 blocks a cluster, 8 and 16 rows a block
SHAPES = [(1, 1), (16, 2), (17, 3), (40, 4), (100, 5), (128, 3), (129, 2), (200, 4), (256, 5)]


def _check(M, N, precision, bar):
    G, V = case(M, N, max(BATCHES), None, seed=3 * M + N)
    ref = oracle.solve(M, N, G, *R, V, voltages=True)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    xb.set_option("orientation", "columns").set_option("algorithm", "thomas")
    xb.factor(precision)
    for b in BATCHES:
        Vd = torch.from_numpy(V[:b].copy()).cuda()
        I, I2 = (torch.zeros((b, N), dtype=torch.float64, device="cuda") for _ in range(2))
        vW = torch.zeros((b, M, N), dtype=torch.float64, device="cuda")
        vB = torch.zeros_like(vW)
        xb.solve(Vd, I, tol=1e-9)
        xb.solve(Vd, I2, vWL=vW, vBL=vB, tol=1e-9)
        xb.sync()
        assert rel_err(I.cpu().numpy(), ref["I"][:b]) <= bar, b
        assert rel_err(I2.cpu().numpy(), ref["I"][:b]) <= bar, b
        assert rel_err(vW.cpu().numpy(), ref["vWL"][:b]) <= bar, b
        assert rel_err(vB.cpu().numpy(), ref["vBL"][:b]) <= bar, b
        if precision == "fp64":
            xb.solve_noalloc(Vd, I2.zero_())
            xb.sync()
            assert torch.equal(I, I2)  # the same kernel on another scratch
    xb.destroy()


@pytest.mark.parametrize("M,N", SHAPES)
def test_few_fp64(M, N):
    _check(M, N, "fp64", 1e-10)  # the suite's bar for FP64


@pytest.mark.parametrize("M,N", SHAPES)
def test_few_mixed(M, N):
    _check(M, N, "fp32_ir", 1e-8)  # and for refined results

