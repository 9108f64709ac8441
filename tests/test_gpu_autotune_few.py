"""The batch autotuner and tiles with few vectors: the automatic choice (clusters) is timed beside the
panel kernels, kept where it is the fastest, and choices of files that do not know it are made again."""
import json

import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = (1.0, 2.5, 2.5, 10.0)
M, N, B = 128, 96, 1


def _tuned(path, maps):
    b = xbar.Batch([(torch.from_numpy(G).cuda(), *R) for G, _ in maps])
    b.autotune("fp32_ir", [B] * len(maps), str(path))
    Vs = [torch.from_numpy(V).cuda() for _, V in maps]
    Is = [torch.zeros((B, N), dtype=torch.float64, device="cuda") for _ in maps]
    b.run("fp32_ir", Vs, Is, tol=1e-9)
    for (G, V), I in zip(maps, Is):  # 1e-8: the suite's bar for refined currents
        assert rel_err(I.cpu().numpy(), oracle.solve(M, N, G, *R, V)["I"]) <= 1e-8
    b.destroy()
    return json.load(open(path))


def test_few_vectors_keep_the_clusters(tmp_path):
    """One vector of 128 rows: the clusters take half of the panels' time (0.54 against 0.96 ms at 128 columns)."""
    path = tmp_path / "tune.json"
    maps = [case(M, N, B, None, seed=t) for t in range(2)]
    key = f"M={M},N={N},B={B},prec=1"
    v = _tuned(path, maps)[key]
    assert v["few"] == 1 and 0 < v["few_ms"] <= min(t for t in v["sweep_ms"] if t > 0)
    assert v["sweep"] in (0, 1) and v["factor"] in (0, 1)
    again = _tuned(path, maps)[key]
    assert again == v  # served from the file
    path.write_text('{\n  "%s": {"sweep": 1, "factor": 1, "orient": -1, "sweep_ms": [0.1, 0.1]}\n}\n' % key)
    assert _tuned(path, maps)[key]["few"] == 1


def test_wide_tiles_have_no_clusters(tmp_path):
    b = xbar.Batch([(torch.from_numpy(case(M, N, 1, None, seed=t)[0]).cuda(), *R) for t in range(2)])
    b.autotune("fp32_ir", [500, 500], str(tmp_path / "tune.json"))
    v = json.load(open(tmp_path / "tune.json"))[f"M={M},N={N},B=500,prec=1"]
    assert v["few"] == 0 and v["few_ms"] == -1
    b.destroy()
