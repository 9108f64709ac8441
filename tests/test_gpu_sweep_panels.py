"""Tensor-core substitutions of large batches: two blocks on an SM (blocks of up to 128 rows) with grids
of more than one round, panels that are not full, one and two elimination chains, and tiles that share
the device."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = (1.0, 2.5, 2.5, 10.0)


# 1e-8 is the suite's bar for refined currents; node voltages follow the same certificate
@pytest.mark.parametrize("M,N,B", [(33, 2, 4930), (100, 5, 4865), (128, 3, 9800), (128, 1, 9729)])
def test_large_batches(M, N, B):
    G, V = case(M, N, B, None, seed=M + N)
    rows = np.unique(np.concatenate([np.arange(0, B, 97), np.arange(B - 70, B)]))
    ref = oracle.solve(M, N, G, *R, V[rows], voltages=True)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    xb.set_option("orientation", "columns").set_option("algorithm", "thomas")
    xb.factor("fp32_ir")
    I = torch.zeros((B, N), dtype=torch.float64, device="cuda")
    vW = torch.zeros((B, M, N), dtype=torch.float64, device="cuda")
    vB = torch.zeros_like(vW)
    xb.solve(torch.from_numpy(V).cuda(), I, vWL=vW, vBL=vB, tol=1e-9)
    assert rel_err(I.cpu().numpy()[rows], ref["I"]) <= 1e-8
    assert rel_err(vW.cpu().numpy()[rows], ref["vWL"]) <= 1e-8
    assert rel_err(vB.cpu().numpy()[rows], ref["vBL"]) <= 1e-8
    xb.destroy()


def test_tiles_side_by_side():
    shapes = [(128, 4, 200), (100, 3, 65), (40, 2, 64), (129, 2, 130)]
    tiles = [case(M, N, B, None, seed=M) for M, N, B in shapes]
    b = xbar.Batch([(torch.from_numpy(G).cuda(), *R) for G, _ in tiles])
    Vs = [torch.from_numpy(V).cuda() for _, V in tiles]
    Is = [torch.zeros((B, N), dtype=torch.float64, device="cuda") for _, N, B in shapes]
    for _ in range(2):  # the first run also captures
        for I in Is:
            I.zero_()
        b.run("fp32_ir", Vs, Is, tol=1e-9, max_iter=6)
        for (M, N, B), (G, V), I in zip(shapes, tiles, Is):
            assert rel_err(I.cpu().numpy(), oracle.solve(M, N, G, *R, V)["I"]) <= 1e-8


# tiles of a batch take the FP64 factor with eight rows a worker block; 1e-10 is the suite's FP64 bar
def test_fp64_tiles_side_by_side():
    shapes = [(16, 9, 3), (32, 17, 64), (33, 20, 5), (100, 51, 65), (128, 65, 20), (130, 66, 9), (256, 129, 4)]
    tiles = [case(M, N, B, None, seed=M) for M, N, B in shapes]
    b = xbar.Batch([(torch.from_numpy(G).cuda(), *R) for G, _ in tiles])
    Vs = [torch.from_numpy(V).cuda() for _, V in tiles]
    Is = [torch.zeros((B, N), dtype=torch.float64, device="cuda") for _, N, B in shapes]
    b.run("fp64", Vs, Is)
    for (M, N, B), (G, V), I in zip(shapes, tiles, Is):
        assert rel_err(I.cpu().numpy(), oracle.solve(M, N, G, *R, V)["I"]) <= 1e-10


def test_row_blocked_tile_new_conductances():
    """A batch with a tile blocked over rows replays its graph; the graph mirrors the tile's current map."""
    shapes = [(96, 20, 65), (40, 32, 64)]
    b = xbar.Batch([(torch.from_numpy(case(M, N, B, None, seed=M)[0]).cuda(), *R) for M, N, B in shapes])
    Vs = [torch.from_numpy(case(M, N, B, None, seed=M)[1]).cuda() for M, N, B in shapes]
    Is = [torch.zeros((B, N), dtype=torch.float64, device="cuda") for _, N, B in shapes]
    Gs = [case(M, N, B, None, seed=M)[0] for M, N, B in shapes]
    for k in range(4):
        if k == 2:  # the row-blocked tile only: the graph is replayed with its new map
            Gs[0] = case(96, 20, 65, None, seed=7)[0]
            xbar._check(xbar.load().xbar_set_conductances(b.tile_handle(0), xbar._ptr(torch.from_numpy(Gs[0]).cuda())))
            torch.cuda.synchronize()
        b.run("fp64", Vs, Is)
        for (M, N, B), G, V, I in zip(shapes, Gs, Vs, Is):
            assert rel_err(I.cpu().numpy(), oracle.solve(M, N, G, *R, V.cpu().numpy())["I"]) <= 1e-10
