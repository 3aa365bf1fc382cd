"""FP64 local solves on both sides of their dispatch: a lane per row (one band
tile, more than two subdomains per SM at one column, four at two to four) and
row pairs, up to eight modes and more."""

import numpy as np
import pytest

from oracle import OracleAMS, csr_to_scipy
from workloads import make_small_2d, make_small_3d

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04864_gb300 import AmsSolver  # noqa: E402

CASES = {
    "few_one_tile": lambda: make_small_2d(side=48, bs=6, m=4, std=1.5, seed=91),             # 64 subdomains
    "some_one_tile": lambda: make_small_2d(side=80, bs=4, m=3, std=1.5, seed=92),            # 400
    "many_one_tile": lambda: make_small_2d(side=133, bs=5, m=4, std=1.5, seed=93, ny=127),   # 702, ragged
    "many_one_tile_10_modes": lambda: make_small_2d(side=104, bs=4, m=10, std=1.5, seed=94),  # 676
    "two_tiles": lambda: make_small_3d(side=15, bs=8, m=4, std=1.5, seed=95),
}


@pytest.fixture(scope="module", params=list(CASES))
def case(request):
    w = CASES[request.param]()
    o = OracleAMS(csr_to_scipy(w.rowptr, w.colind, w.vals), w.part, w.nparts, w.m)
    r = np.random.default_rng(96).standard_normal((5, w.n))
    return w, r, np.stack([o.apply(v) for v in r])


# 1e-10 of the largest entry: the bound of the repository's other FP64 apply tests
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5])
def test_apply_matches_oracle(case, nrhs):
    w, r, ref = case
    s = AmsSolver(w.rowptr, w.colind, w.vals, w.part, w.nparts, w.m, precision="fp64", autotune=False)
    for depth in (0, 1, 3):
        if depth:
            s.set_launch_shape(nrhs, depth=depth)
        z = np.reshape(s.apply_preconditioner(r[:nrhs]), (nrhs, w.n))
        assert np.abs(z - ref[:nrhs]).max() <= 1e-10 * np.abs(ref[:nrhs]).max(), depth
