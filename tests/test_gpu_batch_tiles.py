"""Direct calls on the tiles of a batch (xbar_batch_tile) between runs of its graph: calls that move the
buffers the graph points into or change what it relies on, in both blockings and precisions.  Every run
is compared with the oracle (1e-10 is the suite's bar for FP64, 1e-8 for refined results)."""
import ctypes

import pytest

import oracle
from paper_2410_19993_gb300 import xbar
from tests.gpu_common import case, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = (1.0, 2.5, 2.5, 10.0)
# the first tile is blocked over rows in FP64 (its mirror is solved by cyclic reduction), the second over columns
SHAPES = [(96, 20, 65), (40, 32, 64)]


def _dev(a):
    return torch.from_numpy(a).cuda()


class Tiles:
    def __init__(self, precision, shapes=SHAPES):
        self.precision, self.bar, self.shapes = precision, 1e-10 if precision == "fp64" else 1e-8, shapes
        self.maps = [case(M, N, B, None, seed=M + N) for M, N, B in shapes]
        self.b = xbar.Batch([(_dev(G), *R) for G, _ in self.maps])
        self.V = [_dev(V) for _, V in self.maps]
        self.I = [torch.zeros((B, N), dtype=torch.float64, device="cuda") for _, N, B in shapes]

    def tile(self, t):
        return self.b.tile_handle(t)

    def run(self):
        for I in self.I:
            I.zero_()
        self.b.run(self.precision, self.V, self.I, tol=1e-9, max_iter=6)
        for (M, N, _), (G, V), I in zip(self.shapes, self.maps, self.I):
            assert rel_err(I.cpu().numpy(), oracle.solve(M, N, G, *R, V)["I"]) <= self.bar

    def solve(self, t, B):
        """xbar_solve on the tile's own handle with B vectors: currents and node voltages."""
        M, N, _ = self.shapes[t]
        V = case(M, N, B, None, seed=B)[1]
        Vd, I = _dev(V), torch.zeros((B, N), dtype=torch.float64, device="cuda")
        vW = torch.zeros((B, M, N), dtype=torch.float64, device="cuda")
        lib = xbar.load()
        xbar._check(lib.xbar_solve(self.tile(t), B, xbar._ptr(Vd), xbar._ptr(I), xbar._ptr(vW), None, 1e-9, 10, None))
        xbar._check(lib.xbar_sync(self.tile(t)))
        ref = oracle.solve(M, N, self.maps[t][0], *R, V, voltages=True)
        assert rel_err(I.cpu().numpy(), ref["I"]) <= self.bar
        assert rel_err(vW.cpu().numpy(), ref["vWL"]) <= self.bar


@pytest.mark.parametrize("precision", ["fp64", "fp32_ir"])
def test_larger_solve_between_runs(precision):
    """A direct solve of more vectors reallocates the tile's workspaces; other memory takes their place."""
    s = Tiles(precision)
    s.run()
    s.run()
    for t in range(len(SHAPES)):
        s.solve(t, 300)
        keep = [torch.full((n,), 1.5, dtype=torch.float64, device="cuda") for n in (1 << 12, 1 << 15, 1 << 18)]
        s.run()
        s.run()
        assert all(bool((k == 1.5).all()) for k in keep)


def test_many_widths_between_runs():
    """Substitution plans of cyclic reduction are kept per batch width, the oldest go first."""
    s = Tiles("fp64")
    s.run()
    for B in (1, 2, 4, 8, 16, 17, 33, 49, 60, 20, 36, 50, 40, 64):
        s.solve(0, B)
    s.run()


@pytest.mark.parametrize("option,values", [("factor_kernel", (0, 1, -1)), ("sweep_kernel", (0, 1, -1)),
                                           ("algorithm", (0, -1)), ("orientation", (0, -1))])
@pytest.mark.parametrize("precision", ["fp64", "fp32_ir"])
def test_options_and_factors_between_runs(precision, option, values):
    """A direct factor with another kernel choice leaves another factor and parameter block behind."""
    s = Tiles(precision)
    s.run()
    lib = xbar.load()
    for v in values:
        for t in range(len(SHAPES)):
            xbar._check(lib.xbar_set_option(s.tile(t), xbar.OPTIONS[option], ctypes.c_int(v)))
            xbar._check(lib.xbar_factor(s.tile(t), xbar.PRECISIONS[precision]))
        s.run()
        s.run()


def test_other_precision_between_runs():
    s = Tiles("fp64")
    s.run()
    for t in range(len(SHAPES)):
        xbar._check(xbar.load().xbar_factor(s.tile(t), xbar.PRECISIONS["fp32_ir"]))
    s.run()
    for t in range(len(SHAPES)):
        s.solve(t, 9)


def test_solve_on_a_tile_after_new_conductances():
    """A run factors a tile's new map: the tile's handle can be solved with afterwards, replayed or not."""
    s = Tiles("fp64")
    s.run()
    s.run()
    for k in range(2):
        for t, (M, N, B) in enumerate(SHAPES):
            s.maps[t] = (case(M, N, B, None, seed=100 + 10 * k + t)[0], s.maps[t][1])
            G = _dev(s.maps[t][0])
            torch.cuda.synchronize()
            xbar._check(xbar.load().xbar_set_conductances(s.tile(t), xbar._ptr(G)))
            torch.cuda.synchronize()
            s.run()
            s.solve(t, 3)
            Geff = torch.zeros((M, N), dtype=torch.float64, device="cuda")
            xbar._check(xbar.load().xbar_transfer_matrix(s.tile(t), 1e-9, 10, xbar._ptr(Geff), None))
            assert rel_err((s.V[t] @ Geff).cpu().numpy(), oracle.solve(M, N, s.maps[t][0], *R, s.maps[t][1])["I"]) <= 1e-10


def test_run_follows_the_work_queued_on_a_tile():
    """set_conductances from device memory returns before the tile's stream has stored the map; the next run,
    a replay of the row-blocked tile's graph on another stream, uses the last map set."""
    M, N, B = 256, 100, 4
    s = Tiles("fp64", [(M, N, B)])
    lib, old = xbar.load(), _dev(case(M, N, 1, None, seed=5)[0])
    xbar._check(lib.xbar_set_option(s.tile(0), xbar.OPTIONS["eager_assembly"], 1))  # makes each call longer
    s.run()
    for k in range(3):
        s.run()
        G = case(M, N, 1, None, seed=20 + k)[0]
        s.maps[0] = (G, s.maps[0][1])
        new = _dev(G)
        torch.cuda.synchronize()
        for _ in range(150):  # a queue on the tile's stream that outlasts the run's start
            lib.xbar_set_conductances(s.tile(0), xbar._ptr(old))
        xbar._check(lib.xbar_set_conductances(s.tile(0), xbar._ptr(new)))
    s.run()
