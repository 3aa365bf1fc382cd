"""The tensor-core local solve at the edges of its dispatch: every number of
band tiles per block row (1, 2 and the general path from 3), column counts
below, at and between the eight of an MMA, ring depths around the number of
block rows, both basis types, more than eight modes, and the single vector
that is too long for the one-vector kernel."""

import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

from oracle import OracleAMS, csr_to_scipy
from workloads import make_small_2d, make_small_3d

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04864_gb300 import AmsSolver  # noqa: E402

# name: (workload, band tiles of its widest subdomain)
CASES = {
    "one_tile": (lambda: make_small_2d(side=37, bs=9, m=3, std=1.5, seed=71), 1),
    "two_tiles": (lambda: make_small_3d(side=15, bs=8, m=5, std=1.5, seed=72), 2),
    "two_tiles_ragged": (lambda: make_small_2d(side=61, bs=41, m=4, std=1.5, seed=73, ny=47), 2),
    "three_tiles": (lambda: make_small_3d(side=13, bs=9, m=4, std=1.5, seed=74), 3),
    "three_tiles_12_modes": (lambda: make_small_3d(side=10, bs=9, m=12, std=1.5, seed=75), 3),
    # four tiles a block row only without a coarse space: the eigenproblems' FP64 staging ends at three
    "four_tiles_no_modes": (lambda: make_small_3d(side=11, bs=11, m=0, std=1.5, seed=76), 4),
}


@pytest.fixture(scope="module", params=list(CASES))
def case(request):
    w, c = CASES[request.param][0](), CASES[request.param][1]
    A = csr_to_scipy(w.rowptr, w.colind, w.vals)
    rng = np.random.default_rng(7)
    oracles = {p: OracleAMS(A, w.part, w.nparts, w.m, basis_round=r)
               for p, r in (("fp32", "fp32"), ("fp32_bf16", "bf16"))}
    r = rng.standard_normal((32, w.n))
    return w, c, oracles, r


# FP32 arithmetic of the apply against FP64: 5e-5 of the largest entry, the
# bound of the repository's other apply tests
@pytest.mark.parametrize("prec", ["fp32", "fp32_bf16"])
@pytest.mark.parametrize("nrhs", [2, 3, 8, 9, 32])
def test_apply_matches_oracle(case, prec, nrhs):
    w, c, oracles, r = case
    s = AmsSolver(w.rowptr, w.colind, w.vals, w.part, w.nparts, w.m, precision=prec, autotune=False,
                  coarse=w.m > 0)
    assert s.info()["max_band_tiles"] == c
    ref = np.stack([oracles[prec].apply(r[k]) for k in range(nrhs)])
    shapes = [(2, 0), (6, 8 if nrhs >= 8 else 0)] + ([(3, 16)] if nrhs >= 9 else [])
    for depth, nr in shapes:
        if 4096 * c * (depth + 1) <= 160 * 1024:
            s.set_launch_shape(nrhs, depth=depth, nr=nr)
        z = s.apply_preconditioner(r[:nrhs])
        assert np.abs(z - ref).max() <= 5e-5 * np.abs(ref).max(), (depth, nr)


def test_single_vector_longer_than_the_one_vector_kernel_holds():
    """46,080 rows in one subdomain: 1440 block rows of y exceed the one-vector
    kernel's shared memory.  A Laplacian plus twice the identity has condition
    number 5, so 1440 chained FP32 steps stay within 1e-5."""
    ny, nx = 720, 64
    T = sp.diags([-np.ones(nx - 1), 2 * np.ones(nx), -np.ones(nx - 1)], [-1, 0, 1])
    U = sp.diags([-np.ones(ny - 1), 2 * np.ones(ny), -np.ones(ny - 1)], [-1, 0, 1])
    A = (sp.kron(sp.identity(ny), T) + sp.kron(U, sp.identity(nx)) + 2 * sp.identity(nx * ny)).tocsr()
    A.sort_indices()
    s = AmsSolver(A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data, np.zeros(A.shape[0], np.int32), 1, 0,
                  precision="fp32", autotune=False)
    r = np.random.default_rng(8).standard_normal(A.shape[0])
    z = s.apply_preconditioner(r)
    ref = spla.spsolve(A.tocsc(), r)
    assert np.abs(z - ref).max() <= 1e-5 * np.abs(ref).max()
    z2 = s.apply_preconditioner(np.stack([r, 2 * r]))
    assert np.abs(z2[1] - 2 * ref).max() <= 2e-5 * np.abs(ref).max()
