"""Cyclic reduction with few input vectors: the matrix-vector products of every panel width (1, 2, 4, 8,
16 and the first wide one), the product tiles at blocks of 16 to 256 rows, and the row-blocked solve that
stops at the first block (currents only) beside the one that recovers every node."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = (1.0, 2.5, 2.5, 10.0)


def _run(M, N, precision, options, batches, bar):
    """bar: the suite's bars, 1e-10 for FP64 and 1e-8 for refined currents and voltages."""
    G, V = case(M, N, max(batches), None, seed=M * 7 + N)
    ref = oracle.solve(M, N, G, *R, V, voltages=True)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    for k, v in options.items():
        xb.set_option(k, v)
    xb.factor(precision)
    for b in batches:
        Vd = torch.from_numpy(V[:b].copy()).cuda()
        I = torch.zeros((b, N), dtype=torch.float64, device="cuda")
        I2 = torch.zeros_like(I)
        vW = torch.zeros((b, M, N), dtype=torch.float64, device="cuda")
        vB = torch.zeros_like(vW)
        xb.solve(Vd, I, tol=1e-9)
        xb.solve(Vd, I2, vWL=vW, vBL=vB, tol=1e-9)
        xb.sync()
        assert rel_err(I.cpu().numpy(), ref["I"][:b]) <= bar, (b, "currents only")
        assert rel_err(I2.cpu().numpy(), ref["I"][:b]) <= bar, (b, "with voltages")
        assert rel_err(vW.cpu().numpy(), ref["vWL"][:b]) <= bar
        assert rel_err(vB.cpu().numpy(), ref["vBL"][:b]) <= bar
    xb.destroy()


@pytest.mark.parametrize("M,N", [(5, 1), (16, 2), (33, 17), (128, 3), (130, 9), (256, 4)])
@pytest.mark.parametrize("precision,bar", [("fp64", 1e-10), ("fp32_ir", 1e-8)])
def test_columns_few_vectors(M, N, precision, bar):
    _run(M, N, precision, {"algorithm": "cr", "orientation": "columns"}, [1, 2, 3, 5, 16, 17], bar)


@pytest.mark.parametrize("M,N", [(40, 3), (64, 32), (100, 20), (200, 70)])
@pytest.mark.parametrize("algorithm", ["cr", "thomas"])
def test_rows_first_block_only(M, N, algorithm):
    _run(M, N, "fp64", {"algorithm": algorithm, "orientation": "rows"}, [1, 7, 16, 20], 1e-10)
