"""Launches per phase that the profile reports, for each form of a block-Thomas substitution: an input vector's
and each correction's one (single chain), two (two chains) or three (clusters for few vectors) launches."""
import pytest

from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,B,sweep,each", [
    (16, 9, 700, "tc", 1),     # 16 rows: one chain, one launch of both parts
    (16, 70, 700, "tc", 2),    # longer: two launches
    (16, 9, 5, "simt", 1),     # narrow CUDA-core panels
    (40, 9, 700, "tc", 2),     # two chains
    (40, 3, 700, "tc", 1),     # few columns: one chain
    (130, 3, 700, "tc", 2),    # blocks of more than 128 rows: two launches
    (40, 9, 5, None, 3),       # clusters
])
def test_sweep_launches(M, N, B, sweep, each, monkeypatch):
    if sweep:
        monkeypatch.setenv("XBAR_SWEEP", sweep)
    G, V = case(M, N, B, None, seed=M)
    xb = xbar.Crossbar.assemble(torch.from_numpy(G).cuda(), 1.0, 2.5, 2.5, 10.0)
    xb.set_option("orientation", "columns").set_option("algorithm", "thomas")
    xb.factor("fp32_ir")
    I = torch.zeros((B, N), dtype=torch.float64, device="cuda")
    xb.profile_enable()
    _, info = xb.solve(torch.from_numpy(V).cuda(), I, tol=1e-9)
    assert xb.profile_read()["sweep"]["launches"] == each * (1 + info["iters"])
    xb.destroy()
