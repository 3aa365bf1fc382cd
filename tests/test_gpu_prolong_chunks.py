"""The prolongation from 8 right-hand sides takes a block's subdomains in chunks
of up to 16: blocks with one, with many and with more than a chunk of
subdomains, modes that load by entries, pairs and whole words, more than eight
modes, every basis type."""

import numpy as np
import pytest

from oracle import OracleAMS, csr_to_scipy, pcg
from workloads import make_small_2d, make_small_3d

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_04864_gb300 import AmsBatchedSolver  # noqa: E402

COPIES = 48


# iterations within 2 and solutions within 1e-10 (FP64) or 1e-6 of the oracle's:
# the bounds of the repository's other batched tests
@pytest.mark.parametrize("prec", ["fp32_bf16", "fp32", "fp64"])
@pytest.mark.parametrize("m,nrhs", [(3, 8), (6, 9), (8, 8), (8, 32), (12, 17)])
def test_blocks_of_many_subdomains(prec, m, nrhs):
    ws = [make_small_2d(side=24, bs=4, m=m, std=1.5, seed=81),          # 36 subdomains
          make_small_2d(side=19, bs=5, m=m, std=1.5, seed=82, ny=26),   # 24, ragged
          make_small_3d(side=9, bs=4, m=m, std=1.5, seed=83)]           # 27, down to one row
    systems = [(w.rowptr, w.colind, w.vals, w.part, w.nparts, w.m) for w in ws] * COPIES
    rhs = [np.random.default_rng(84 + i).standard_normal((nrhs, w.n)) for i, w in enumerate(ws)]
    b = AmsBatchedSolver(systems, precision=prec, autotune=False)
    shape = (1, 2, 4)                                   # blocks per SM: about one to four a system
    refs = []
    for i, w in enumerate(ws):
        A = csr_to_scipy(w.rowptr, w.colind, w.vals)
        o = OracleAMS(A, w.part, w.nparts, w.m, basis_round={"fp32_bf16": "bf16", "fp32": "fp32"}.get(prec))
        refs.append([pcg(A, rhs[i][k], o.apply, rtol=1e-8) for k in (0, nrhs - 1)])
    tol = 1e-10 if prec == "fp64" else 1e-6
    for bps in shape:
        b.set_launch_shape(nrhs, bps_sub=bps)
        u, its, _ = b.solve(b.pack(rhs * COPIES), nrhs, rtol=1e-8)
        us = b.unpack(u, nrhs)
        for s in (0, 1, 2, 3 * COPIES - 3, 3 * COPIES - 2, 3 * COPIES - 1):
            for j, k in enumerate((0, nrhs - 1)):
                ref = refs[s % 3][j]
                assert abs(int(its[s, k]) - ref.iters) <= 2, (bps, s, k)
                assert np.linalg.norm(us[s][k] - ref.u) <= tol * np.linalg.norm(ref.u), (bps, s, k)
