"""Surrogate predictions run part of their work beside the line model on a second stream: alternating maps
and batch sizes through one surrogate give, bit for bit, what a fresh one gives for each."""
import pytest

from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = (1.0, 2.5, 2.5, 10.0)


def predict(s, G, V):
    I = torch.zeros((V.shape[0], G.shape[1]), dtype=torch.float64, device="cuda")
    err = torch.zeros_like(I)
    s.predict(G, V, I, err_est=err)
    return I, err


@pytest.mark.parametrize("M,N", [(33, 20), (128, 128), (200, 150)])
def test_alternating_maps(M, N):
    def make():
        return xbar.Surrogate(M, N, R, passes=2, g_scale=1e-4, v_scale=0.5, seed=3)
    work = []
    for k, B in enumerate((1, 300, 65)):
        G, V = case(M, N, B, None, seed=k)
        work.append((torch.from_numpy(G).cuda(), torch.from_numpy(V).cuda()))
    want = [predict(make(), G, V) for G, V in work]
    s = make()
    for _ in range(10):
        for (G, V), (I0, e0) in zip(work, want):
            I, err = predict(s, G, V)
            assert torch.equal(I, I0) and torch.equal(err, e0)
