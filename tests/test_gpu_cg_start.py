"""Start vectors of the solvers: the zero start skips the operator of the first residual, a
nonzero one (also of only one right-hand side of a batch) does not."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from gpu_helpers import launches, make_case  # noqa: E402
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


@pytest.mark.parametrize("eo", [False, True], ids=["cg", "eo"])
@pytest.mark.parametrize("mode", [dw.DW_F64, dw.DW_F32])
def test_one_zero_start_of_a_batch_skips_nothing(mode, eo):
    # RHS 0 starts at zero, RHS 1 at its solution: if the batch were taken for a zero start,
    # the first residual of RHS 1 would be its right-hand side and it would iterate
    dims, Ls, mfs = (4, 4, 4, 8), 6, [0.1, 0.2]
    U, rhs = make_case(dims, Ls, 2, seed=33)
    lat = Lattice(dims, Ls, prec=dw.DW_F64)
    lat.load_gauge(U)
    solve = lat.solve_eo if eo else lat.cg
    x, b = lat.empty(2).zero_(), lat.pack(rhs)
    assert solve(x, b, mfs, nrhs=2, tol=1e-10, mode=mode)[0] == dw.DW_OK
    sol = x.clone()
    x[: lat.fermion_bytes(1)].zero_()
    status, stats = solve(x, b, mfs, nrhs=2, tol=1e-8, mode=mode)
    assert status == dw.DW_OK
    assert stats[0].iters > 0 and stats[1].iters == 0
    if not eo:  # (the even-odd solve forms the even sites anew)
        assert torch.equal(x[lat.fermion_bytes(1):], sol[lat.fermion_bytes(1):])
    lat.close()


@pytest.mark.parametrize("eo,hops", [(False, 2), (True, 4)], ids=["cg", "eo"])
def test_zero_start_skips_the_first_operator(eo, hops):
    # against a start so small that it changes no bit of the residual: the same solve, with
    # the FP64 D and D^+ (two hops each in the even-odd operators) of one more residual
    dims, Ls = (4, 4, 4, 8), 6
    U, rhs = make_case(dims, Ls, 1, seed=34)
    lat = Lattice(dims, Ls, prec=dw.DW_F64)
    lat.load_gauge(U)
    solve = lat.solve_eo if eo else lat.cg
    b, stats = lat.pack(rhs), {}
    x = lat.empty().view(torch.float64)

    def run(start):
        x.fill_(start)
        stats[start] = solve(x, b, 0.1, tol=1e-8, mode=dw.DW_F32)

    run(0.0)  # tunes
    n = [launches(lambda s=s: run(s), "dslash_kernel<dw::F64") for s in (0.0, 1e-30)]
    assert n[1] - n[0] == hops and n[0] > 0
    assert stats[0.0][0] == stats[1e-30][0] == dw.DW_OK
    assert stats[0.0][1][0].iters == stats[1e-30][1][0].iters
    lat.close()
