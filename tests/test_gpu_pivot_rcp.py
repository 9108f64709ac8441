"""The FP64 pivot reciprocal (common.cuh) against 1 / x.  Its error is at most 0.5 + 2^-7 units in the last
place, so it differs from the correctly rounded quotient by one unit at most, and only where 1 / x lies within
2^-7 units of the middle between two numbers: about one input in 64.  Outside its exponent window it divides."""
import numpy as np
import pytest

from tests.kernel_probe import compile_probe, ptr

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = """
#include "common.cuh"
__global__ void rcp_kernel(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = xbar::pivot_rcp(x[i]);
}
extern "C" int rcp(const double* x, double* y, int n) {
  rcp_kernel<<<(n + 255) / 256, 256>>>(x, y, n);
  return cudaDeviceSynchronize() ? 1 : 0;
}
"""


@pytest.fixture(scope="module")
def rcp(tmp_path_factory):
    lib = compile_probe(tmp_path_factory.mktemp("rcp"), "rcp", SOURCE)

    def call(x):
        x = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()
        y = torch.zeros_like(x)
        torch.cuda.synchronize()
        assert lib.rcp(ptr(x), ptr(y), x.numel()) == 0
        return y.cpu().numpy()
    return call


def _units(y, x):
    """Distance of y from 1 / x in representable numbers (positive, finite values)."""
    return np.abs(y.view(np.int64) - (1.0 / x).view(np.int64))


def test_random_pivots(rcp):
    rng = np.random.default_rng(0)
    n = 1 << 21
    x = rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(-950, 950, n)
    d = _units(rcp(x), x)
    assert d.max() <= 1
    assert np.mean(d > 0) <= 1.5 / 64  # the expected 1/64 and half of it for the bound's rough first bits


def test_edges_of_the_window(rcp):
    m = np.concatenate([[1.0, np.nextafter(2.0, 1.0), 1.5, np.nextafter(1.0, 2.0)],
                        np.random.default_rng(1).uniform(1.0, 2.0, 500)])
    for e in (-1022, -960, -959, -958, 0, 959, 960, 961, 1022, 1023):  # biased 64 .. 1983 is the window
        x = m * 2.0 ** (e / 2) * 2.0 ** (e - e / 2) if e % 2 == 0 else m * 2.0 ** ((e - 1) / 2) * 2.0 ** ((e + 1) / 2)
        y = rcp(x)
        d = _units(y, x)
        inside = -959 <= e <= 960
        assert d.max() <= (1 if inside else 0), e
    x = np.array([5e-324, 1e-310, 2.2e-308, 1.7e308, 0.0, -0.0, np.inf, -np.inf])
    with np.errstate(divide="ignore", over="ignore"):
        assert np.array_equal(rcp(x), 1.0 / x)
    assert np.isnan(rcp(np.array([np.nan]))).all()
    x = -np.random.default_rng(2).uniform(1.0, 2.0, 1000)
    assert np.array_equal(rcp(x), -rcp(-x))
