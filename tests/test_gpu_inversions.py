"""Accuracy of the FP32 block inversions (Gauss-Jordan, no pivoting) against 64 bits.

Yardstick: the same inversion one pivot at a time with FP32 rounding, emulated here.  Handling a pair of
pivots by its 2 x 2 determinant instead rounds once more and errs 1.74 to 1.87 times as much (emulated),
so the bar is 1.35 times the emulated error: half way, in the logarithm, between the two."""
import numpy as np
import pytest

from tests.kernel_probe import compile_probe, ptr

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BAR = 1.35
SEEDS = range(6)


def _round(x):
    return np.asarray(x, dtype=np.float64).astype(np.float32).astype(np.float64)


def _emulated(Z):
    """Scalar sweeps with fused multiply-adds: every operation in FP64, rounded to FP32."""
    A = Z.copy()
    for q in range(A.shape[0]):
        c, inv = A[:, q].copy(), _round(1.0 / A[q, q])
        f = _round(A[q] * inv)
        f[q] = inv
        A[:, q] = 0.0
        A = _round(A - c[:, None] * f[None, :])
        A[q] = f
    return A


def _error(X, Z):
    ref = np.linalg.inv(Z)
    return np.linalg.norm(X - ref) / np.linalg.norm(ref)


def _block(n, rng):
    """A symmetric M-matrix coupled as weakly as the equilibrated column blocks of a crossbar of 1e-6 to 1e-4 S
    behind wires of a few ohm: (off-diagonal part, grounded row sums), exact in FP32, and so are the sums of
    the off-diagonal part."""
    off = -np.triu(rng.integers(0, 4096, (n, n)) * 2.0 ** -40, 1)
    return off + off.T, rng.integers(1 << 20, 1 << 22, n) * 2.0 ** -20


def _matrix(off, rowsum):
    return off + np.diag(_round(rowsum - off.sum(1)))


GJ = """
#include "gemm_jobs.cu"
extern "C" int gj32(const float* src, float* dst, int n, void* job) {
  const xbar::GjJob<float> j{src, dst, n, n};
  if (cudaMemcpy(job, &j, sizeof(j), cudaMemcpyHostToDevice)) return 1;
  if (xbar::launch_gj_inverse<float>((const xbar::GjJob<float>*)job, 1, n, nullptr, 0)) return 2;
  return cudaDeviceSynchronize() ? 3 : 0;
}
"""


def test_panel_inversion(tmp_path):
    """The 8-row panels of cyclic reduction's inversions: sizes at and between its three thread layouts."""
    lib = compile_probe(tmp_path, "gj", GJ)
    job = torch.zeros(64, dtype=torch.uint8, device="cuda")
    for n in (16, 32, 48, 64, 112, 128):
        err = ref = 0.0
        for s in SEEDS:
            Z = _matrix(*_block(n, np.random.default_rng(s)))
            src = torch.from_numpy(Z.astype(np.float32)).cuda()
            dst = torch.zeros_like(src)
            torch.cuda.synchronize()
            assert lib.gj32(ptr(src), ptr(dst), n, ptr(job)) == 0
            err += _error(dst.cpu().numpy().astype(np.float64), Z)
            ref += _error(_emulated(Z), Z)
        assert err <= BAR * ref, (n, err, ref)


CLUSTER = """
#include <string.h>
#include "factor_cluster.cu"
// a crossbar of one column: X = (off + the grounded diagonal)^-1
extern "C" int cluster32(int n, const float* off, const double* h, const float* ones, float* X, float* work, void* par,
                         unsigned* status) {
  xbar::FactorParams<float> p;
  memset(&p, 0, sizeof(p));
  p.M = p.Mp = n;
  p.N = 1;
  p.gw = 1.0;
  p.Coff = off;
  p.h = h;
  p.X = X;
  p.s32 = ones;
  p.e32 = ones;
  p.sig = work;
  p.pbuf = work + 4 * n;
  if (cudaMemcpy(par, &p, sizeof(p), cudaMemcpyHostToDevice)) return 1;
  if (xbar::launch_factor_cluster((const xbar::FactorParams<float>*)par, n, 1, 0, status, 0)) return 2;
  return cudaDeviceSynchronize() ? 3 : 0;
}
extern "C" int cluster_work_floats(int n) { return 4 * n + (int)xbar::factor_cluster_pbuf_floats(n); }
"""


def test_cluster_inversion(tmp_path):
    """The pivot blocks of the cluster factor (two to sixteen blocks a cluster)."""
    lib = compile_probe(tmp_path, "cluster", CLUSTER)
    for n in (32, 48, 64, 128, 144, 256):
        err = ref = 0.0
        for s in SEEDS:
            off, rowsum = _block(n, np.random.default_rng(s))
            Z = _matrix(off, rowsum)
            X = torch.zeros((n, n), dtype=torch.float32, device="cuda")
            work = torch.zeros(lib.cluster_work_floats(n), dtype=torch.float32, device="cuda")
            par = torch.zeros(512, dtype=torch.uint8, device="cuda")
            st = torch.zeros(4, dtype=torch.int32, device="cuda")
            dev = [torch.from_numpy(a).cuda() for a in (off.astype(np.float32), rowsum, np.ones(n, dtype=np.float32))]
            torch.cuda.synchronize()
            assert lib.cluster32(n, *[ptr(d) for d in dev], ptr(X), ptr(work), ptr(par), ptr(st)) == 0
            assert int(st[0]) == 0
            err += _error(X.cpu().numpy().astype(np.float64), Z)
            ref += _error(_emulated(Z), Z)
        assert err <= BAR * ref, (n, err, ref)
