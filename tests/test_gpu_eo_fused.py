"""Dhat and Dhat^+ at the sizes where the A^-1 step fused into the hop can go wrong: one
slice, odd Ls, the most slice groups that fit a CTA and one more (the separate pass), planes
that do not fill a tile, several right-hand sides."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from oracle import eo  # noqa: E402
from gpu_helpers import BC, TOL, make_case  # noqa: E402
from paper_2112_01852_gb300 import dw  # noqa: E402
from paper_2112_01852_gb300.lattice import Lattice  # noqa: E402


@pytest.mark.parametrize("prec", [dw.DW_F32, dw.DW_F16], ids=["f32", "f16"])
@pytest.mark.parametrize("dims,Ls,kind", [
    ((4, 2, 4, 2), 1, dw.DW_MOBIUS), ((6, 6, 2, 4), 2, dw.DW_MOBIUS),
    ((4, 4, 2, 6), 7, dw.DW_MOBIUS), ((10, 2, 2, 4), 9, dw.DW_SHAMIR),
    ((8, 10, 2, 2), 16, dw.DW_MOBIUS), ((4, 6, 2, 2), 18, dw.DW_MOBIUS)])
def test_schur_edges(dims, Ls, kind, prec):
    U, psi = make_case(dims, Ls, 2, seed=61, links="haar")
    mf = [0.02, 0.3]
    b, c = (1.5, 0.5) if kind == dw.DW_MOBIUS else (1.0, 0.0)
    lat = Lattice(dims, Ls, kind=kind, prec=prec)
    lat.load_gauge(U)
    _, odd = lat.pack_eo(psi)
    x = eo.project(lat.unpack(lat.pack(psi), 2), dims, 1)
    zero = lat.empty_eo(2).zero_()
    for dag, f in ((0, eo.schur), (1, eo.schur_dag)):
        out = lat.empty_eo(2)
        dw.dw_apply_schur(lat.handle, out.data_ptr(), odd.data_ptr(), mf, 2, dag)
        got = lat.unpack_eo(zero, out, 2)
        for r in range(2):
            ref = f(x[r:r + 1], U, dims, Ls, 1.8, b, c, [mf[r]], BC)
            assert oracle.rel_l2(got[r:r + 1], ref) <= TOL[prec], (dag, r)
    lat.close()
