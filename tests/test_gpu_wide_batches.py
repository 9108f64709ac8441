"""Batches so wide that one column block holds more than 2^31 values (rows times vectors): the row-blocked
FP64 solve by cyclic reduction of two blocks, whose right-hand side and forward reduction run over both."""
import numpy as np
import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_more_than_2_31_values_a_block():
    M, N = 2, 16
    B = (1 << 31) // N + 1000
    need = 8 * B * (3 * M * N + M + N + M)  # the substitution's three arrays, V, I and the mirror's currents
    if torch.cuda.mem_get_info()[0] < need + (8 << 30):
        pytest.skip("needs %d GB of free device memory" % (need >> 30))
    R = (1.0, 2.5, 2.5, 10.0)
    G, V = case(M, N, 4096, None, seed=3)
    ref = oracle.solve(M, N, G, *R, V)["I"]
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), *R)
    xb.set_option("orientation", "rows")
    xb.factor("fp64")
    Vd = torch.from_numpy(V).cuda().repeat((B + 4095) // 4096, 1)[:B].contiguous()
    I = torch.zeros((B, N), dtype=torch.float64, device="cuda")
    xb.solve(Vd, I)
    xb.sync()
    for b in (0, B // 3 // 4096 * 4096, (B - 1) // 4096 * 4096):
        n = min(4096, B - b)
        assert rel_err(I[b:b + n].cpu().numpy(), ref[:n]) <= 1e-10  # the suite's bar for FP64
    xb.destroy()
    del Vd, I
    torch.cuda.empty_cache()
