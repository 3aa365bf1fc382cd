"""The local solve of up to four right-hand sides (and of one on a subdomain too
long for the one-vector kernel): as close to the 64-bit solution as plain FP32
substitution, every split of the columns over warps, and its launch count."""

import numpy as np
import pytest
import scipy.linalg as la
import scipy.sparse as sp

from oracle import OracleAMS, csr_to_scipy
from workloads import make_small_2d, make_small_3d

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04864_gb300 import AmsError, AmsSolver  # noqa: E402


def _grid(nx, ny, shift):
    """Five-point Laplacian plus shift on ny lines of nx cells: band width nx in this order."""
    def lap(n):
        return sp.diags([-np.ones(n - 1), 2 * np.ones(n), -np.ones(n - 1)], [-1, 0, 1])
    A = (sp.kron(sp.identity(ny), lap(nx)) + sp.kron(lap(ny), sp.identity(nx)) + shift * sp.identity(nx * ny)).tocsr()
    A.sort_indices()
    return A


def _solver(A, part=None, nparts=1, **kw):
    part = np.zeros(A.shape[0], np.int32) if part is None else part
    return AmsSolver(A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data, part, nparts, 0, precision="fp32",
                     autotune=False, **kw)


# One subdomain without a coarse space: the preconditioner is the local solve.  The bound is twice the error of LAPACK's
# banded substitution in FP32 with the factor rounded to FP32, which is what "plain FP32" gives on the same system.
@pytest.mark.parametrize("nx,ny,nrhs", [(32, 96, 2), (32, 96, 3), (32, 96, 4), (64, 50, 2), (64, 50, 4), (90, 70, 2),
                                        (90, 70, 3), (64, 720, 1), (64, 720, 2)])
@pytest.mark.parametrize("kind", ["random", "constant"])
def test_as_accurate_as_plain_fp32(nx, ny, nrhs, kind):
    A = _grid(nx, ny, 0.5)
    n = A.shape[0]
    r = np.random.default_rng(5).standard_normal((nrhs, n)) if kind == "random" else np.ones((nrhs, n))
    ab = np.zeros((nx + 1, n))
    for k in range(nx + 1):
        ab[k, :n - k] = A.diagonal(-k)
    L = la.cholesky_banded(ab, lower=True)
    exact = la.cho_solve_banded((L, True), r.T).T
    plain = la.cho_solve_banded((L.astype(np.float32), True), r.T.astype(np.float32)).T
    assert plain.dtype == np.float32
    z = np.reshape(_solver(A).apply_preconditioner(r), (nrhs, n))
    for k in range(nrhs):
        assert np.linalg.norm(z[k] - exact[k]) <= 2 * np.linalg.norm(plain[k] - exact[k]), k


CASES = {
    "one_tile": lambda: make_small_2d(side=37, bs=9, m=3, std=1.5, seed=71),
    "two_tiles": lambda: make_small_3d(side=15, bs=8, m=5, std=1.5, seed=72),
    "three_tiles_12_modes": lambda: make_small_3d(side=10, bs=9, m=12, std=1.5, seed=75),
}


# 5e-5 of the largest entry: the bound of the repository's other FP32 apply tests
@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("prec", ["fp32", "fp32_bf16"])
def test_column_splits_match_oracle(name, prec):
    w = CASES[name]()
    o = OracleAMS(csr_to_scipy(w.rowptr, w.colind, w.vals), w.part, w.nparts, w.m,
                  basis_round="fp32" if prec == "fp32" else "bf16")
    r = np.random.default_rng(6).standard_normal((4, w.n))
    ref = np.stack([o.apply(v) for v in r])
    s = AmsSolver(w.rowptr, w.colind, w.vals, w.part, w.nparts, w.m, precision=prec, autotune=False)
    for nrhs, nr in ((2, 0), (2, 2), (3, 2), (3, 4), (4, 0), (4, 2), (4, 4)):
        for depth in (0, 2, 3, 6):
            if depth:
                s.set_launch_shape(nrhs, depth=depth, nr=nr)
            z = s.apply_preconditioner(r[:nrhs])
            assert np.abs(z - ref[:nrhs]).max() <= 5e-5 * np.abs(ref[:nrhs]).max(), (nrhs, nr, depth)


def test_launch_count_with_two_band_widths():
    """One vector on a subdomain too long for the one-vector kernel takes a launch per band width, as two do."""
    A = sp.block_diag([_grid(64, 720, 2.0), _grid(1, 40, 2.0)]).tocsr()
    A.sort_indices()
    part = (np.arange(A.shape[0]) >= 64 * 720).astype(np.int32)
    s = _solver(A, part, 2)
    r = np.random.default_rng(7).standard_normal((2, A.shape[0]))
    counts = []
    for nrhs in (1, 2):
        before = s.info()["kernel_launches"]
        s.apply_preconditioner(r[:nrhs])
        counts.append(s.info()["kernel_launches"] - before)
    assert counts[0] == counts[1] == 5   # two permutes, two band widths, the prolongation


@pytest.mark.parametrize("nrhs", [2, 4])
def test_exhausted_wait_reports_timeout_and_the_next_handle_solves(nrhs):
    """Every block first waits, for a short budget, on a barrier that nothing completes."""
    w = make_small_2d(side=48, bs=8, m=3, std=1.5, seed=78)
    f = np.random.default_rng(9).standard_normal((nrhs, w.n))
    args = (w.rowptr, w.colind, w.vals, w.part, w.nparts, w.m)
    s = AmsSolver(*args, precision="fp32", autotune=False, spin_budget_cycles=20000, timeout_probe=True)
    with pytest.raises(AmsError) as e:
        s.apply_preconditioner(f)
    assert e.value.status == 5   # AMS_ERR_DEVICE_TIMEOUT
    u, _, rel = AmsSolver(*args, precision="fp32", autotune=False).solve(f)
    assert (rel <= 1e-8).all()
