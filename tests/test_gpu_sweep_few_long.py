"""Few-vector substitutions on clusters along chains of many steps: the ring of factor slices wraps around
(three or four slices) and the exchange's two phases alternate, for every panel width, rows-per-block
choice and precision, in direct solves, tile batches (whose passes skip) and row-blocked solves (first block
only)."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = (1.0, 2.5, 2.5, 10.0)
# (M, N, batches of 1, 2, 4 and 8 vectors a panel): 8 and 16 rows a block, three and four slices in the ring
SHAPES = [(17, 23, (1, 30, 70, 200)), (40, 21, (3, 20, 40, 100)), (100, 20, (1, 10, 17, 40)),
          (129, 21, (2, 9, 20, 50)), (256, 24, (1, 7, 15, 30))]


# 1e-10 and 1e-8 are the suite's bars
@pytest.mark.parametrize("precision,bar", [("fp64", 1e-10), ("fp32_ir", 1e-8)])
@pytest.mark.parametrize("M,N,batches", SHAPES)
def test_long_chains(M, N, batches, precision, bar):
    G, V = case(M, N, max(batches), None, seed=M)
    ref = oracle.solve(M, N, G, *R, V, voltages=True)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    xb.set_option("orientation", "columns").set_option("algorithm", "thomas")
    xb.factor(precision)
    for b in batches:
        Vd = torch.from_numpy(np.ascontiguousarray(V[:b])).cuda()
        I = torch.zeros((b, N), dtype=torch.float64, device="cuda")
        vW = torch.zeros((b, M, N), dtype=torch.float64, device="cuda")
        xb.solve(Vd, I, tol=1e-9)
        xb.sync()
        assert rel_err(I.cpu().numpy(), ref["I"][:b]) <= bar, b
        xb.solve(Vd, I, vWL=vW, tol=1e-9)
        xb.sync()
        assert rel_err(vW.cpu().numpy(), ref["vWL"][:b]) <= bar, b
    xb.destroy()


@pytest.mark.parametrize("precision,bar", [("fp64", 1e-10), ("fp32_ir", 1e-8)])
def test_long_chains_in_a_batch(precision, bar):
    shapes = [(M, N, b[1]) for M, N, b in SHAPES]
    maps = [case(M, N, B, None, seed=M) for M, N, B in shapes]
    b = xbar.Batch([(torch.from_numpy(G).cuda(), *R) for G, _ in maps])
    for t in range(len(maps)):
        xbar._check(xbar.load().xbar_set_option(b.tile_handle(t), xbar.OPTIONS["orientation"], 0))
    Vs = [torch.from_numpy(V).cuda() for _, V in maps]
    Is = [torch.zeros((B, N), dtype=torch.float64, device="cuda") for _, N, B in shapes]
    for _ in range(2):
        b.run(precision, Vs, Is, tol=1e-9, max_iter=6)
        for (M, N, _), (G, V), I in zip(shapes, maps, Is):
            assert rel_err(I.cpu().numpy(), oracle.solve(M, N, G, *R, V)["I"]) <= bar
    b.destroy()


def test_first_block_only():
    """Row-blocked block Thomas (mirrors of 17 to 64 rows), currents alone: the outward part stops at the first block."""
    for M, N, B in [(60, 17, 3), (90, 40, 20), (140, 64, 1)]:
        G, V = case(M, N, B, None, seed=M)
        xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
        xb.set_option("orientation", "rows").set_option("algorithm", "thomas")
        xb.factor("fp64")
        I = torch.zeros((B, N), dtype=torch.float64, device="cuda")
        xb.solve(torch.from_numpy(V).cuda(), I)
        xb.sync()
        assert rel_err(I.cpu().numpy(), oracle.solve(M, N, G, *R, V)["I"]) <= 1e-10
        xb.destroy()
