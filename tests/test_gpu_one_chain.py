"""Substitutions of a factor with a single elimination chain, both parts in one launch (tensor-core panels of
blocks of up to 128 rows, narrow CUDA-core panels): two to many columns, ragged rows, full and ragged
panels, currents alone and with node voltages; and factors of maps with few columns, which take one chain."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = (1.0, 2.5, 2.5, 10.0)


# 1e-8 is the suite's bar for refined results
def _check(M, N, batches):
    G, V = case(M, N, max(batches), None, seed=2 * M + N)
    ref = oracle.solve(M, N, G, *R, V, voltages=True)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    xb.set_option("orientation", "columns").set_option("algorithm", "thomas")
    xb.factor("fp32_ir")
    for b in batches:
        Vd = torch.from_numpy(np.ascontiguousarray(V[:b])).cuda()
        I, I2 = (torch.zeros((b, N), dtype=torch.float64, device="cuda") for _ in range(2))
        vW = torch.zeros((b, M, N), dtype=torch.float64, device="cuda")
        vB = torch.zeros_like(vW)
        xb.solve(Vd, I, tol=1e-9)
        xb.solve(Vd, I2, vWL=vW, vBL=vB, tol=1e-9)
        assert rel_err(I.cpu().numpy(), ref["I"][:b]) <= 1e-8, b
        assert rel_err(I2.cpu().numpy(), ref["I"][:b]) <= 1e-8, b
        assert rel_err(vW.cpu().numpy(), ref["vWL"][:b]) <= 1e-8, b
        assert rel_err(vB.cpu().numpy(), ref["vBL"][:b]) <= 1e-8, b
    xb.destroy()


@pytest.mark.parametrize("sweep", ["tc", "simt"])
@pytest.mark.parametrize("M,N", [(16, 2), (33, 5), (100, 20), (128, 33)])
def test_group_factor(M, N, sweep, monkeypatch):
    monkeypatch.setenv("XBAR_FACTOR", "group")
    monkeypatch.setenv("XBAR_SWEEP", sweep)
    _check(M, N, [1, 5, 64, 65, 300])


@pytest.mark.parametrize("M,N", [(32, 2), (100, 3), (129, 4), (256, 3)])
def test_few_columns(M, N):
    _check(M, N, [1, 40, 700])


def test_crowded_tiles():
    """Tiles that fill the device: one chain, no clusters for few vectors, FP64 factors of 32 rows by one block."""
    for precision, bar in (("fp32_ir", 1e-8), ("fp64", 1e-10)):
        for M, N, B in [(32, 12, 3), (32, 8, 65), (16, 5, 2), (16, 5, 40)]:
            T = 56
            maps = [case(M, N, B, None, seed=t) for t in range(T)]
            b = xbar.Batch([(torch.from_numpy(G).cuda(), *R) for G, _ in maps])
            for t in range(T):
                xbar._check(xbar.load().xbar_set_option(b.tile_handle(t), xbar.OPTIONS["orientation"], 0))
            Vs = [torch.from_numpy(V).cuda() for _, V in maps]
            Is = [torch.zeros((B, N), dtype=torch.float64, device="cuda") for _ in maps]
            for _ in range(2):
                b.run(precision, Vs, Is, tol=1e-9, max_iter=6)
            for (G, V), I in zip(maps, Is):
                assert rel_err(I.cpu().numpy(), oracle.solve(M, N, G, *R, V)["I"]) <= bar
            b.destroy()
