"""The FP64 factor's plan (kernels.h) fits the device it is made for: a cooperative launch of more blocks
than the SMs can hold is an error, so with fewer SMs the plan narrows and then gives way to the group kernel."""
import ctypes

import pytest

from tests.kernel_probe import compile_probe

SOURCE = """
#include "kernels.h"
extern "C" void plan(int Mp, int N, int nsm, int beside, int* out) {
  const xbar::Factor64Plan f = xbar::factor64_plan(Mp, N, nsm, beside != 0);
  out[0] = f.rows;
  out[1] = f.meet;
  out[2] = f.rows ? xbar::factor64_blocks(Mp, N, f) : 0;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    lib = compile_probe(tmp_path_factory.mktemp("plan"), "plan", SOURCE)

    def call(*args):
        out = (ctypes.c_int * 3)()
        lib.plan(*args, out)
        return tuple(out)
    return call


def test_plans_fit(plan):
    for Mp in range(16, 1025, 16):
        for N in (1, 2, 3, 64):
            for beside in (0, 1):
                for nsm in (1, 2, 4, 7, 16, 20, 33, 66, 76, 129, 130, 148, 152):
                    rows, meet, blocks = plan(Mp, N, nsm, beside)
                    if rows == 0:
                        # one chain of 8-row workers does not fit either
                        assert (1 if Mp == 16 else Mp // 8 + 1) > nsm
                        continue
                    assert 1 <= blocks <= nsm and 0 <= meet < N
                    assert rows == 8 or (rows == 4 and Mp <= 256) or (rows == 2 and Mp <= 128)


def test_plans_of_a_whole_device(plan):
    """152 SMs: every size has a plan, two chains up to 512 rows."""
    for Mp in range(16, 1025, 16):
        rows, meet, _ = plan(Mp, 64, 152, 0)
        assert rows == (2 if Mp <= 128 else 4 if Mp <= 256 else 8)
        assert meet == (31 if Mp <= 512 else 63)
        assert plan(Mp, 64, 152, 1)[0] == 8
