"""The prolongation takes the backward coarse block, and the x update, only at
the right-hand-side strides whose kernels are compiled with them.  No launch:
the calls have no subdomains."""

from .native import build_native, run_native

SOURCE = r"""
#include <cstdio>
#include "launch.h"
using namespace ams;
int main() {
    double there = 0.0;
    for (int ld = 1; ld <= 32; ld *= 2)
        for (int qmat = 0; qmat < 2; ++qmat)
            for (int x = 0; x < 2; ++x) {
                LaunchCtx L{};
                L.ld = ld;
                ProlongArgs a{};
                a.mmax = 8;
                a.mode = 2;
                a.qmat = qmat ? &there : nullptr;
                a.x = x ? &there : nullptr;
                std::printf("%d %d %d %d\n", ld, qmat, x,
                            launch_prolong_update(L, AMS_PREC_FP32, a) == cudaErrorInvalidValue);
            }
}
"""


def test_strides_without_the_code_refuse_the_arguments(tmp_path):
    got = {tuple(map(int, line.split())) for line in run_native(build_native(tmp_path, SOURCE))}
    assert got == {(ld, q, x, int((q and ld > 4) or (not x and ld < 8)))
                   for ld in (1, 2, 4, 8, 16, 32) for q in (0, 1) for x in (0, 1)}
