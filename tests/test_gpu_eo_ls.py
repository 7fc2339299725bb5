"""The Ls that the even-odd operators and the solve take, and those that they refuse: FP64
operators with their adjoints or not at all; FP32 / FP16 up to 16 slice groups (Dhat a third
or a half of its groups).  A refused call launches nothing: `out` stays as it is."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from oracle import eo  # noqa: E402
from gpu_helpers import BC, TOL, make_case  # noqa: E402
from paper_2112_01852_gb300 import dw  # noqa: E402
from paper_2112_01852_gb300.lattice import Lattice  # noqa: E402

DIMS = (4, 2, 2, 4)


@pytest.mark.parametrize("prec,dag,taken,refused", [
    (dw.DW_F64, 0, (7, 9, 16, 21, 64), (11, 22, 34)),
    (dw.DW_F64, 1, (7, 9, 16, 21, 64), (11, 22, 34)),
    (dw.DW_F32, 0, (15, 32, 36, 33), (17, 34, 38, 80)), (dw.DW_F32, 1, (15, 32), (17, 34, 36)),
    (dw.DW_F16, 0, (36,), (34,)), (dw.DW_F16, 1, (32,), (36,))])
def test_schur_ls_limits(prec, dag, taken, refused):
    for Ls in taken + refused:
        U, _ = make_case(DIMS, 1, 1, seed=3)
        lat = Lattice(DIMS, Ls, prec=prec)
        lat.load_gauge(U)
        x, y = lat.empty_eo().zero_(), lat.empty_eo().fill_(1)

        def schur():
            dw.dw_apply_schur(lat.handle, y.data_ptr(), x.data_ptr(), [0.1], 1, dag,
                              torch.cuda.current_stream().cuda_stream)

        if Ls in taken:
            schur()
            torch.cuda.synchronize()
            assert not y.any()
        else:
            with pytest.raises(dw.DWError) as e:
                schur()
            assert e.value.code == dw.DW_ERR_ARG, Ls
            torch.cuda.synchronize()
            assert bool((y == 1).all()), Ls
        lat.close()


@pytest.mark.parametrize("mode", [dw.DW_F64, dw.DW_F32])
@pytest.mark.parametrize("Ls,ok", [(9, True), (20, True), (11, False), (30, False)])
def test_solve_ls_limits(Ls, ok, mode):
    U, psi = make_case(DIMS, Ls, 1, seed=4)
    lat = Lattice(DIMS, Ls, prec=dw.DW_F64)
    lat.load_gauge(U)
    eta, x = lat.pack(psi), lat.empty().zero_()
    if ok:
        assert lat.solve_eo(x, eta, 0.2, mode=mode)[0] == dw.DW_OK
    else:
        with pytest.raises(dw.DWError) as e:
            lat.solve_eo(x, eta, 0.2, mode=mode)
        assert e.value.code == dw.DW_ERR_ARG
        assert not x.any()
    lat.close()


@pytest.mark.parametrize("Ls", [9, 18, 21])
def test_fp64_schur_over_several_ctas(Ls):
    # more slice groups than one FP64 CTA holds: Dhat^+ as a cluster
    U, psi = make_case(DIMS, Ls, 1, seed=5, links="haar")
    lat = Lattice(DIMS, Ls, prec=dw.DW_F64)
    lat.load_gauge(U)
    _, odd = lat.pack_eo(psi)
    x = eo.project(psi, DIMS, 1)
    zero = lat.empty_eo().zero_()
    for dag, f in ((0, eo.schur), (1, eo.schur_dag)):
        out = lat.empty_eo()
        dw.dw_apply_schur(lat.handle, out.data_ptr(), odd.data_ptr(), [0.05], 1, dag)
        ref = f(x, U, DIMS, Ls, 1.8, 1.5, 0.5, [0.05], BC)
        assert oracle.rel_l2(lat.unpack_eo(zero, out), ref) <= TOL[dw.DW_F64], dag
    lat.close()
