"""The setup's host loops run in chunks on several threads: the first faulty row
is the one reported, whichever chunk finds its fault first, and systems of
several chunks, with rows longer than the fixed buffer, give what the oracle
gives."""

import numpy as np
import pytest
import scipy.sparse as sp

from oracle import OracleAMS, pcg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04864_gb300 import AmsSolver  # noqa: E402


def _chain(n):
    A = sp.diags([-np.ones(n - 1), np.full(n, 2.5), -np.ones(n - 1)], [-1, 0, 1]).tocsr()
    A.sort_indices()
    return A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data.copy()


def _asymmetric(rp, ci, v, row):
    v[rp[row] + 2] *= 1.5                        # the entry right of the diagonal


def _nonpositive(rp, ci, v, row):
    v[rp[row] + 1] = -1.0


def _unsorted(rp, ci, v, row):
    for w in (ci, v):                            # diagonal and right neighbour, with their values
        w[rp[row] + 1], w[rp[row] + 2] = w[rp[row] + 2], w[rp[row] + 1]


def _column(rp, ci, v, row):
    ci[rp[row] + 2] = 2 ** 30


def _pointer(rp, ci, v, row):
    rp[row + 1] = rp[row] - 1


FAULTS = {_asymmetric: "not symmetric at \\({0}, {1}\\)", _nonpositive: "non-positive diagonal in row {0}",
          _unsorted: "columns not strictly ascending in row {0}", _column: "column index out of range in row {0}",
          _pointer: "rowptr decreases at row {0}"}


@pytest.mark.parametrize("later", list(FAULTS), ids=lambda f: f.__name__)
@pytest.mark.parametrize("first", list(FAULTS), ids=lambda f: f.__name__)
def test_first_faulty_row_is_reported(first, later):
    n = 100_000                                   # twelve chunks of rows
    rp, ci, v = _chain(n)
    part = (np.arange(n) // 500).astype(np.int32)
    row = 40_000
    later(rp, ci, v, 90_000)
    first(rp, ci, v, row)
    with pytest.raises(Exception, match=FAULTS[first].format(row, row + 1)):
        AmsSolver(rp, ci, v, part, n // 500, 2)


def test_many_chunks_and_long_rows_match_oracle():
    """A chain of 70,000 rows (8 chunks of rows, 2 of the 141 subdomains) whose rows
    1000 + 10000 j also couple to 98 rows before them, in two subdomains."""
    n = 70_000
    A = sp.diags([-np.ones(n - 1), -np.ones(n - 1)], [-1, 1]).tolil()
    for j in range(1000, n, 10_000):
        for i in range(j - 99, j - 1):
            A[j, i] = A[i, j] = -0.25
    A = A.tocsr()
    A = (A + sp.diags(0.5 - np.asarray(A.sum(axis=1)).ravel())).tocsr()
    A.sort_indices()
    part = ((np.arange(n) + 50) // 500).astype(np.int32)
    # Gershgorin: eigenvalues in [0.5, 53.5], and both solves stop at 1e-8
    tol = 2 * 107 * 1e-8
    f = np.random.default_rng(9).standard_normal(n)
    s = AmsSolver(A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data, part, int(part.max()) + 1, 2,
                  precision="fp64", autotune=False)
    ref = pcg(A, f, OracleAMS(A, part, int(part.max()) + 1, 2).apply, rtol=1e-8)
    u, its, _ = s.solve(f, rtol=1e-8)
    assert abs(int(np.ravel(its)[0]) - ref.iters) <= 2
    assert np.linalg.norm(np.ravel(u) - ref.u) <= tol * np.linalg.norm(ref.u)
