"""Start vectors of the solvers: the zero start skips the operator of the first residual, a
nonzero one (also of only one right-hand side of a batch) does not."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from gpu_helpers import make_case  # noqa: E402
from paper_2112_01852_gb300 import dw  # noqa: E402
from paper_2112_01852_gb300.lattice import Lattice  # noqa: E402


@pytest.mark.parametrize("mode", [dw.DW_F64, dw.DW_F32])
@pytest.mark.parametrize("starts", [(0.0, 0.0), (0.0, 1.0), (2.0, 1.0)])
def test_cg_start_vectors(mode, starts):
    dims, Ls, mfs = (4, 4, 4, 8), 6, [0.1, 0.2]
    U, rhs = make_case(dims, Ls, 2, seed=31)
    _, guess = make_case(dims, Ls, 2, seed=32)
    lat = Lattice(dims, Ls, prec=dw.DW_F64)
    lat.load_gauge(U)
    x = lat.pack(np.stack([starts[r] * guess[r] for r in range(2)]))
    status, stats = lat.cg(x, lat.pack(rhs), mfs, nrhs=2, tol=1e-10, maxit=5000, mode=mode)
    assert status == dw.DW_OK
    got = lat.unpack(x, 2)
    for r in range(2):
        Ax = oracle.dwdagdw(got[r:r + 1], U, dims, Ls, 1.8, 1.5, 0.5, [mfs[r]])
        assert oracle.rel_l2(Ax, rhs[r:r + 1]) <= 1e-10
    # at the solution the first residual already meets a looser tol: no iteration
    status, stats = lat.cg(x, lat.pack(rhs), mfs, nrhs=2, tol=1e-9, maxit=5000, mode=mode)
    assert status == dw.DW_OK and all(s.iters == 0 for s in stats)
    lat.close()
