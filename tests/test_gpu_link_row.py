"""The third row of an FP32 link, rebuilt as conj(row0 x row1): its rounding error.

Dhop of a source with one nonzero component copies a link's column exactly (projection and
sum add zeros), so the rows a kernel works with can be read from its output, the rebuilt one
among them."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2112_01852_gb300 import dw  # noqa: E402
from paper_2112_01852_gb300.lattice import Lattice  # noqa: E402

DIMS = (16, 8, 8, 4)


def _links(eps):
    """exp(i eps H), H Hermitian, traceless, Gaussian."""
    rng = np.random.RandomState(1)
    n = int(np.prod(DIMS)) * 4
    a = rng.randn(n, 3, 3) + 1j * rng.randn(n, 3, 3)
    h = (a + a.conj().transpose(0, 2, 1)) / 2
    h -= np.trace(h, axis1=1, axis2=2)[:, None, None] / 3 * np.eye(3)
    w, v = np.linalg.eigh(h)
    u = (v * np.exp(1j * eps * w)[:, None, :]) @ v.conj().transpose(0, 2, 1)
    return np.ascontiguousarray(u.reshape(-1, 4, 3, 3))


@pytest.mark.parametrize("variant", [None, 0, 1, 4], ids=["untuned", "v0", "v1", "v4"])
@pytest.mark.parametrize("eps", [0.0, 0.03, 0.1])
def test_rebuilt_row_rounds_once_at_size_one(eps, variant):
    # Re row2_2 of a link near one is Re(a_0 b_1) of order one less three terms of order eps
    # or smaller.  Added smallest first, it is off by half a unit in the last place of the
    # result and by the roundings of the three partial sums below it, each at most
    # 2^-24 (|t2| + |t3| + |t4|).
    U = _links(eps)
    lat = Lattice(DIMS, 1, prec=dw.DW_F32)
    lat.load_gauge(U)
    if variant is not None:
        lat.set_tile(dw.DW_OP_DHOP, 1, 32, variant)
    t, z, y, x = (k.reshape(-1) for k in np.indices(DIMS[::-1]))
    for off in (1, 2, 3):  # sources four sites apart: no neighbour in common
        at = np.where((x % 4 == off) & (y % 4 == off) & (z % 4 == off) & (t % 4 == off))[0]
        rows = np.zeros((len(at), 3, 3), complex)
        for col in range(3):
            psi = np.zeros((1, lat.V4, 1, 4, 3), complex)
            psi[0, at, 0, 0, col] = 1.0
            out = lat.empty(1)
            lat.dhop(out, lat.pack(psi))
            rows[:, :, col] = lat.unpack(out)[0, at - 1, 0, 0]  # U_x(at - 1) of the hop to at - 1
        a, b, got = rows[:, 0], rows[:, 1], rows[:, 2]
        assert np.abs(a - U[at - 1, 0, 0]).max() <= 2.0 ** -24  # the stored row
        ref = np.cross(a, b).conj()
        assert np.abs(got - ref).max() <= 1.5e-7
        small = (np.abs(a[:, 0].imag * b[:, 1].imag) + np.abs(a[:, 1].real * b[:, 0].real) +
                 np.abs(a[:, 1].imag * b[:, 0].imag))
        bound = 0.5 * np.spacing(np.abs(ref[:, 2].real).astype(np.float32)) + 3 * 2.0 ** -24 * small
        assert np.all(np.abs(got[:, 2].real - ref[:, 2].real) <= bound)
    lat.close()
