"""Ring depths that the tuner tries for the FP64 local solve: up to six where a
lane per row runs (left-looking), three where row pairs do, each with its own
kernel's shared memory.  Host code only."""

import pytest

from .native import build_native, run_native

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "launch.h"
using namespace ams;
int main(int, char** argv) {
    LocalSolveArgs a{};
    a.cmax = std::atoi(argv[1]);
    a.ncols = std::atoi(argv[2]);
    for (a.ld = 1; a.ld < a.ncols;) a.ld *= 2;
    a.mmax = std::atoi(argv[3]);
    a.sms = 100;
    for (a.nsub = 50; a.nsub <= 750; a.nsub += 100)
        std::printf("%d %d %zu\n", a.nsub, local_solve_max_depth(a), local_solve_launch_smem(a, 2));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    return build_native(tmp_path_factory.mktemp("native"), SOURCE)


# from how many subdomains an SM (100 SMs) a lane per row runs; None: never
@pytest.mark.parametrize("cmax,ncols,mmax,line", [(1, 1, 8, 2), (1, 2, 8, 3), (1, 3, 8, 4), (1, 4, 8, 4), (1, 1, 9, 1),
                                                  (1, 2, 16, 3), (1, 3, 12, 2), (1, 4, 12, 2), (1, 5, 8, None),
                                                  (2, 1, 8, None), (2, 4, 12, None)])
def test_depths_follow_the_kernel(program, cmax, ncols, mmax, line):
    row = 8 * (1024 * cmax + 32)      # a block row of the factor, pivots included
    ld = 1 << (ncols - 1).bit_length()
    rows = (cmax + 3) * row + 8 * ((cmax + 1) * 32 * ld + 32 * ld)
    pairs = 3 * row + 8 * (2 * cmax + 1) * 32 * ncols
    for text in run_native(program, cmax, ncols, mmax):
        nsub, depth, smem = map(int, text.split())
        by_rows = line is not None and nsub > 100 * line
        assert (depth, smem) == ((6, rows) if by_rows else (3, pairs)), nsub
