"""dw_apply_host reports a bounded wait that gave up: with an untuned tile (the rule takes the
row-staged variant for these), in slabs and in one piece.  wait_polls = 0 gives up the first
wait of each step at once; the second one lets the copies land, so the output is right."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from gpu_helpers import TOL, make_case, max_rel, run_oracle  # noqa: E402
from paper_2112_01852_gb300 import dw  # noqa: E402
from paper_2112_01852_gb300.lattice import Lattice  # noqa: E402


# 32 x 32 x 8 sites a time slice: slabs of one slice; 16 x 16 x 6 x 8: one piece
@pytest.mark.parametrize("dims,Ls,prec,op", [
    ((32, 32, 8, 4), 8, dw.DW_F32, dw.DW_OP_DHOP), ((32, 32, 8, 4), 8, dw.DW_F16, dw.DW_OP_DDAGD),
    ((16, 16, 6, 8), 8, dw.DW_F32, dw.DW_OP_DHOP_DAG)])
def test_host_apply_reports_a_wait_that_gave_up(dims, Ls, prec, op):
    U, psi = make_case(dims, Ls, 1, seed=23)
    lat = Lattice(dims, Ls, prec=prec)
    lat.load_gauge(U)
    staged = dw.DW_OP_D if op == dw.DW_OP_DDAGD else op
    assert dw.dw_get_tile(lat.handle, staged, prec, 1)[2] == 6
    x = lat.pack(psi)
    xin = torch.empty(x.numel(), dtype=torch.uint8, pin_memory=True)
    xin.copy_(x)
    out = torch.zeros(x.numel(), dtype=torch.uint8).pin_memory()
    mf = [0.05] if op == dw.DW_OP_DDAGD else None
    ref = run_oracle(op, psi, U, dims, Ls, 1.8, 1.5, 0.5, [0.05])

    def right():
        return max_rel(lat.unpack(out.cuda(), 1), ref) <= TOL[prec]

    for _ in range(2):
        dw.dw_set_wait_polls(lat.handle, 0)
        with pytest.raises(dw.DWError) as e:
            lat.apply_host(op, out, xin, mf)
        assert e.value.code == dw.DW_ERR_TIMEOUT
        assert right()
        dw.dw_set_wait_polls(lat.handle, -1)
        out.zero_()
        lat.apply_host(op, out, xin, mf)  # the word was cleared
        assert right()
        dw.dw_device_status(lat.handle)
    lat.close()
