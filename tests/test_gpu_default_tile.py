"""Untuned tiles: every branch of the rule gives the general path's result (variant 0, one
slice per thread) bit for bit, over precisions, even, odd and prime Ls, ragged planes, one
and several right-hand sides, lattices below and above the small-lattice line."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from gpu_helpers import make_case  # noqa: E402
from paper_2112_01852_gb300 import dw  # noqa: E402
from paper_2112_01852_gb300.lattice import Lattice  # noqa: E402

SHAPES = [((4, 4, 4, 4), 8, 1), ((16, 16, 4, 12), 8, 1), ((16, 16, 4, 12), 12, 2),
          ((24, 24, 4, 6), 16, 1), ((11, 10, 7, 18), 9, 1), ((24, 8, 6, 10), 7, 3),
          ((18, 17, 6, 8), 10, 1), ((26, 16, 6, 4), 10, 1), ((40, 8, 6, 8), 8, 1),
          ((8, 6, 5, 3), 1, 2), ((8, 8, 4, 4), 34, 1), ((6, 8, 4, 4), 26, 2)]


def apply(lt, op, y, x, mf, nrhs):
    if op <= dw.DW_OP_DHOP_DAG:
        lt.dhop(y, x, nrhs, dag=op == dw.DW_OP_DHOP_DAG)
    elif op == dw.DW_OP_D:
        lt.D(y, x, mf, nrhs)
    else:
        lt.Ddag(y, x, mf, nrhs)


@pytest.mark.parametrize("prec", [dw.DW_F64, dw.DW_F32, dw.DW_F16], ids=["f64", "f32", "f16"])
@pytest.mark.parametrize("dims,Ls,nrhs", SHAPES)
def test_default_equals_general_path(dims, Ls, nrhs, prec):
    U, psi = make_case(dims, Ls, nrhs, seed=71)
    mf = [0.01 * (r + 1) for r in range(nrhs)]
    lat, gen = (Lattice(dims, Ls, prec=prec) for _ in range(2))
    x = lat.pack(psi)
    for lt in (lat, gen):
        lt.load_gauge(U)
    for op in (dw.DW_OP_DHOP, dw.DW_OP_DHOP_DAG, dw.DW_OP_D, dw.DW_OP_DDAG):
        done = False
        for spt in (1, 2, 3, 4):  # the smallest that the general path takes
            try:
                gen.set_tile(op, spt, 32, 0)
                done = True
                break
            except dw.DWError:
                continue
        if not done:  # an Ls that the general path refuses is refused untuned too
            with pytest.raises(dw.DWError):
                apply(lat, op, lat.empty(nrhs), x, mf, nrhs)
            continue
        out = []
        for lt in (lat, gen):
            y = lt.empty(nrhs).zero_()
            apply(lt, op, y, x, mf, nrhs)
            out.append(y)
        assert torch.equal(out[0], out[1]), (op, dw.dw_get_tile(lat.handle, op, prec, nrhs))
    for lt in (lat, gen):
        lt.close()
