"""The filtered subspace iteration of the local eigenproblems at the edges of
its rules: block sizes around the modes (fewer dofs than columns, 8 and 9
modes), a shift so small that only plain steps are safe, a large one, and an
iteration cap that ends inside a filter."""

import numpy as np
import pytest
import scipy.linalg as la

from oracle import csr_to_scipy, local_matrices
from workloads import make_small_2d, make_small_3d

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04864_gb300 import AmsSolver  # noqa: E402

CASES = {
    "8_modes": (lambda: make_small_2d(side=40, bs=16, m=8, std=2.0, seed=91, ny=33), {}),
    "9_modes": (lambda: make_small_2d(side=30, bs=15, m=9, std=1.0, seed=92), {}),
    "fewer_dofs_than_columns": (lambda: make_small_3d(side=5, bs=2, m=6, std=1.0, seed=93), {}),
    "tiny_shift": (lambda: make_small_2d(side=24, bs=12, m=5, std=2.0, seed=94), {"eig_shift": 1e-5}),
    "large_shift": (lambda: make_small_2d(side=24, bs=12, m=5, std=2.0, seed=95), {"eig_shift": 1.0}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_eigenpairs_match_lapack(name):
    w, opt = CASES[name][0](), CASES[name][1]
    A = csr_to_scipy(w.rowptr, w.colind, w.vals)
    s = AmsSolver(w.rowptr, w.colind, w.vals, w.part, w.nparts, w.m, precision="fp64", **opt)
    mi, lams, psis = s.coarse_basis()
    # residuals are iterated to 1e-13 in the S^-1 norm with S-orthonormal
    # columns, and bound the eigenvalue error; the repository's other
    # eigenpair test allows 1e-11
    assert s.info()["eig_max_residual"] <= 1e-11
    for i in range(w.nparts):
        _, Ah, sw = local_matrices(A, np.flatnonzero(w.part == i))
        Ah = Ah.toarray() if hasattr(Ah, "toarray") else np.asarray(Ah)
        d = 1.0 / np.sqrt(sw)
        ref = la.eigvalsh(d[:, None] * Ah * d[None, :])[:mi[i]]
        assert np.abs(lams[i] - ref).max() <= 1e-11 * max(1.0, np.abs(ref).max())
        assert np.abs(psis[i].T @ (sw[:, None] * psis[i]) - np.eye(mi[i])).max() <= 1e-11


@pytest.mark.parametrize("cap", [1, 4, 5, 6, 7, 9])
def test_iteration_cap_is_kept(cap):
    w = make_small_2d(side=24, bs=12, m=5, std=2.0, seed=96)
    s = AmsSolver(w.rowptr, w.colind, w.vals, w.part, w.nparts, w.m, precision="fp64", eig_maxit=cap)
    assert s.info()["eig_iterations"] == cap
    mi, lams, psis = s.coarse_basis()
    assert all(np.isfinite(p).all() for p in psis)
