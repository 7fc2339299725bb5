"""Field conversions at the values where rounding can go wrong: ties, carries into the
exponent, the largest and smallest normal numbers, subnormals, zeros, infinities, NaN.
numpy's casts (IEEE round to nearest even) are the reference; the results are exact."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2112_01852_gb300 import dw, inputs  # noqa: E402
from paper_2112_01852_gb300.lattice import Lattice  # noqa: E402


def _specials(n, bits, emin, emax):
    """n doubles around the rounding points of a format with `bits` fraction bits."""
    rng = np.random.RandomState(7)
    e = rng.randint(emin - bits - 3, emax + 3, n)
    frac = rng.randint(0, 1 << bits, n).astype(np.float64) / (1 << bits)
    frac[: n // 8] = 1.0 - 2.0 ** -bits  # all ones: a carry into the exponent
    half = rng.choice([0.0, 0.5, 0.5 - 2.0 ** -20, 0.5 + 2.0 ** -20, 0.25, 0.75], n)
    v = np.ldexp(1.0 + frac + half * 2.0 ** -bits, e) * rng.choice([-1.0, 1.0], n)
    v[:8] = [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, 1.7e308]
    return v


@pytest.mark.parametrize("prec,dt,bits,emin,emax",
                         [(dw.DW_F32, np.float32, 23, -126, 127),
                          (dw.DW_F16, np.float16, 10, -14, 15)])
@pytest.mark.parametrize("dims,Ls", [((4, 4, 4, 4), 8), ((3, 5, 2, 7), 5), ((2, 2, 2, 2), 1)])
def test_pack_unpack_round_as_ieee(dims, Ls, prec, dt, bits, emin, emax):
    lat = Lattice(dims, Ls, prec=prec)
    n = lat.V5 * 24
    psi = _specials(n, bits, emin, emax).view(np.complex128).reshape(1, lat.V4, Ls, 4, 3)
    got = lat.unpack(lat.pack(psi)).view(np.float64)
    with np.errstate(over="ignore", invalid="ignore"):
        ref = psi.view(np.float64).astype(dt).astype(np.float64)
    assert np.array_equal(got, ref, equal_nan=True)
    num = ~np.isnan(ref)
    assert np.array_equal(np.signbit(got[num]), np.signbit(ref[num]))
    lat.close()


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (3, 5, 2, 7)])
@pytest.mark.parametrize("prec", [dw.DW_F64, dw.DW_F32, dw.DW_F16])
def test_load_gauge_copies(dims, prec):
    """Dhop against the oracle reads every stored link, its boundary sign included."""
    import oracle
    U = inputs.haar_su3_field(dims, seed=4)
    psi = inputs.gaussian_fermion(dims, 2, 1, seed=4)
    for bc in ((1, 1, 1, -1), (-1, 1, -1, 1)):
        lat = Lattice(dims, 2, prec=prec, bc=bc)
        lat.load_gauge(U)
        y = lat.empty(1)
        lat.dhop(y, lat.pack(psi))
        ref = oracle.dhop(psi, U, dims, 2, bc)
        # element rounding of the storage type, accumulated over 8 hops
        tol = {dw.DW_F64: 1e-14, dw.DW_F32: 1e-6, dw.DW_F16: 2e-3}[prec]
        assert oracle.rel_l2(lat.unpack(y), ref) < tol
        lat.close()
