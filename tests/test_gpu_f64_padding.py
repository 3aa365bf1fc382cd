"""FP64 calls with a number of right-hand sides between two strides: the local
solves leave zeros in the columns that no right-hand side has, and a handle
that is called with one number after another gives each the oracle's result
(its captured loops are kept per number, its work vectors are shared)."""

import numpy as np
import pytest

from oracle import OracleAMS, csr_to_scipy, pcg
from workloads import make_small_3d

from .native import build_native, run_native

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04864_gb300 import AmsSolver  # noqa: E402

# two subdomains of 40 rows (two block rows, the second ragged), one band tile, factor = identity: z_f = r, r_c = Psi^T r
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <limits>
#include <vector>
#include "launch.h"
using namespace ams;
static double* up(const std::vector<double>& v) {
    double* d = nullptr;
    cudaMalloc(&d, v.size() * sizeof(double));
    cudaMemcpy(d, v.data(), v.size() * sizeof(double), cudaMemcpyHostToDevice);
    return d;
}
int main(int, char** argv) {
    const int ncols = std::atoi(argv[1]), ld = std::atoi(argv[2]), nsub = std::atoi(argv[3]), n = 40, m = 2;
    std::vector<SubInfo> subs(nsub);
    std::vector<double> fac(2 * blockrow_elems(1), 0.0), r(nsub * n * ld, 0.0), psi(nsub * n * m);
    for (int k = 0; k < 2; ++k)
        for (int i = 0; i < 32; ++i) fac[k * blockrow_elems(1) + 1024 + i] = 1.0;
    for (int s = 0; s < nsub; ++s) {
        subs[s] = SubInfo{};
        subs[s].row0 = s * n;
        subs[s].psi_off = s * n * m;
        subs[s].coff = s * m;
        subs[s].n = n;
        subs[s].nb = 2;
        subs[s].c = 1;
        subs[s].m = m;
    }
    for (size_t i = 0; i < psi.size(); ++i) psi[i] = 1.0 + (double)(i % 3);
    for (int i = 0; i < nsub * n; ++i)
        for (int k = 0; k < ncols; ++k) r[i * ld + k] = 1.0 + (i * 7 + k) % 11;
    const double nan = std::numeric_limits<double>::quiet_NaN();
    std::vector<double> zf(r.size(), nan), rc(nsub * m * ld, nan);
    SubInfo* d_subs = nullptr;
    cudaMalloc(&d_subs, nsub * sizeof(SubInfo));
    cudaMemcpy(d_subs, subs.data(), nsub * sizeof(SubInfo), cudaMemcpyHostToDevice);
    double *d_zf = up(zf), *d_rc = up(rc);
    LocalSolveArgs a{};
    a.nsub = nsub;
    a.subs = d_subs;
    a.in.r = up(r);
    a.ld = ld;
    a.cmax = 1;
    a.mmax = m;
    a.ncols = ncols;
    a.sms = 152;
    if (launch_local_solve(a, up(fac), up(psi), d_zf, d_rc) != cudaSuccess) return 1;
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    cudaMemcpy(zf.data(), d_zf, zf.size() * sizeof(double), cudaMemcpyDeviceToHost);
    cudaMemcpy(rc.data(), d_rc, rc.size() * sizeof(double), cudaMemcpyDeviceToHost);
    int bad = 0;
    for (size_t i = 0; i < zf.size(); ++i) bad += !(zf[i] == r[i]);
    for (int i = 0; i < nsub * m; ++i)
        for (int k = 0; k < ld; ++k) {
            double want = 0.0;
            for (int j = 0; j < n; ++j) want += psi[(i / m * n + j) * m + i % m] * r[(i / m * n + j) * ld + k];
            bad += !(rc[i * ld + k] == want);   // whole numbers: exact in any order
        }
    std::printf("%d\n", bad);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    return build_native(tmp_path_factory.mktemp("native"), SOURCE)


# row pairs with every number of lanes a task, and (700 subdomains, up to four columns) a lane per row
@pytest.mark.parametrize("ncols,ld,nsub", [(1, 1, 2), (2, 2, 2), (3, 4, 2), (5, 8, 2), (7, 8, 2), (9, 16, 2), (17, 32, 2),
                                           (31, 32, 2), (32, 32, 2), (3, 4, 700)])
def test_columns_without_a_right_hand_side_are_zero(program, ncols, ld, nsub):
    assert run_native(program, ncols, ld, nsub) == ["0"]


@pytest.mark.parametrize("cycle", [False, True])
def test_one_handle_with_one_count_after_another(cycle):
    w = make_small_3d(side=15, bs=8, m=4, std=1.5, seed=97)
    A = csr_to_scipy(w.rowptr, w.colind, w.vals)
    o = OracleAMS(A, w.part, w.nparts, w.m)
    omega = 1.0 / o.local_lambda_max() if cycle else 0.0
    apply = (lambda v: o.apply_two_grid(v, omega)) if cycle else o.apply
    f = np.random.default_rng(98).standard_normal((8, w.n))
    ref = [pcg(A, v, apply, rtol=1e-8) for v in f]
    s = AmsSolver(w.rowptr, w.colind, w.vals, w.part, w.nparts, w.m, precision="fp64", two_grid_omega=omega)
    for k, nrhs in enumerate((5, 8, 6, 5, 3, 5)):
        if k == 3:   # drops the loops captured for this stride
            s.set_launch_shape(nrhs, depth=1)
        u, its, _ = s.solve(f[:nrhs], rtol=1e-8)
        for i in range(nrhs):
            # the bounds of the repository's other FP64 solves: two iterations, 1e-10 (here between two stops at 1e-8,
            # whose solutions differ by the residual's size when the counts do)
            assert abs(int(its[i]) - ref[i].iters) <= 2
            tol = 1e-10 if int(its[i]) == ref[i].iters else 1e-6
            assert np.linalg.norm(u[i] - ref[i].u) <= tol * np.linalg.norm(ref[i].u)


def test_reported_bytes_are_those_of_the_columns_there_are():
    w = make_small_3d(side=15, bs=8, m=4, std=1.5, seed=97)
    s = AmsSolver(w.rowptr, w.colind, w.vals, w.part, w.nparts, w.m, precision="fp64")
    f = np.random.default_rng(98).standard_normal((8, w.n))
    per_column = 8 * (3 * w.n + s.info()["ncoarse"])   # r and q in, z_f and r_c out
    local = {}
    for nrhs in (8, 5, 7):
        local[nrhs] = s.profile_solve(f[:nrhs])[1]["bytes"]
        assert s.time_kernel(1, 1)[1] == local[nrhs]
    assert local[8] - local[5] == 3 * per_column and local[8] - local[7] == per_column
