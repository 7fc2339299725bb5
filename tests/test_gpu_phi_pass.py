"""The FP64 D with its (b + cK) pass: bit for bit the fused kernel, which a capturing
stream takes (no allocation there), and within the oracle's tolerance."""

import ctypes
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from gpu_helpers import TOL, launches, make_case  # noqa: E402
from paper_2112_01852_gb300 import dw  # noqa: E402
from paper_2112_01852_gb300.lattice import Lattice  # noqa: E402


# V5 nrhs just below and at the 2^15 threshold of the pass, ragged extents, odd Ls, Ls = 1
@pytest.mark.parametrize("dims,Ls,nrhs,kind", [
    ((8, 8, 8, 8), 8, 1, dw.DW_MOBIUS), ((7, 9, 5, 11), 9, 2, dw.DW_MOBIUS),
    ((8, 8, 8, 8), 7, 1, dw.DW_MOBIUS), ((16, 16, 8, 16), 1, 1, dw.DW_MOBIUS),
    ((8, 4, 8, 16), 8, 3, dw.DW_SHAMIR)])
def test_phi_pass_equals_fused(dims, Ls, nrhs, kind):
    U, psi = make_case(dims, Ls, nrhs, 11)
    mfs = [0.01 + 0.02 * r for r in range(nrhs)]
    lat = Lattice(dims, Ls, kind=kind, prec=dw.DW_F64)
    lat.load_gauge(U)
    x = lat.pack(psi)
    y, ref = lat.empty(nrhs), lat.empty(nrhs)
    y.zero_()
    ref.zero_()
    lat.D(y, x, mfs, nrhs)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        lat.D(ref, x, mfs, nrhs)
    ref.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, ref)
    # the pass runs from the threshold on, and not in the captured call
    runs = [launches(f, "phi_kernel") for f in (lambda: lat.D(y, x, mfs, nrhs), graph.replay)]
    assert runs == [1 if lat.V5 * nrhs >= 1 << 15 else 0, 0]
    got = lat.unpack(y, nrhs)
    b, c = (1.5, 0.5) if kind == dw.DW_MOBIUS else (1.0, 0.0)
    want = np.concatenate([oracle.dw(psi[r:r + 1], U, dims, Ls, 1.8, b, c, mfs[r])
                           for r in range(nrhs)])
    assert oracle.rel_l2(got, want) <= TOL[dw.DW_F64]
    lat.close()


@pytest.mark.parametrize("calls", [1, 2])
def test_phi_pass_leaves_another_streams_capture_alone(calls):
    # The first D of a lattice creates its pool and allocates; a capture in progress on
    # another thread (in the global mode, torch's default) must survive that.
    dims, Ls = (8, 8, 8, 16), 8
    U, psi = make_case(dims, Ls, 1, 13)
    lats = [Lattice(dims, Ls, prec=dw.DW_F64) for _ in range(3)]
    for lt in lats:
        lt.load_gauge(U)
    cap, lat, warm = lats
    x = cap.pack(psi)
    y, ref, z = (lat.empty().zero_() for _ in range(3))
    warm.D(ref, x, 0.05)  # loads the kernels, on a lattice of its own
    warm.dhop(z, x)
    torch.cuda.synchronize()
    side, errors = torch.cuda.Stream(), []

    def other():
        try:
            with torch.cuda.stream(side):
                for _ in range(calls):
                    lat.D(y, x, 0.05)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    out = cap.empty().zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cap.dhop(out, x)
        th = threading.Thread(target=other)
        th.start()
        th.join()
    assert not errors
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, ref) and torch.equal(out, z)
    for lt in lats:
        lt.close()


def test_tuner_times_the_phi_pass():
    # the tiles of an FP64 D above the threshold are compared as they run: phi, then the hop
    dims, Ls = (8, 8, 8, 16), 8
    U, _ = make_case(dims, Ls, 1, 14)
    lat = Lattice(dims, Ls, prec=dw.DW_F64)
    lat.load_gauge(U)
    n = launches(lambda: lat.tune(dw.DW_OP_D), "phi_kernel")
    small = Lattice((8, 8, 8, 8), 7, prec=dw.DW_F64)  # below it: the fused kernel
    small.load_gauge(U[: small.V4])
    assert n > 0 and launches(lambda: small.tune(dw.DW_OP_D), "phi_kernel") == 0
    lat.close()
    small.close()


def test_noalloc_ddagd_takes_the_phi_pass():
    # `out` is free until the D^+ pass: the pass needs no allocation there
    dims, Ls = (8, 8, 8, 16), 8
    U, psi = make_case(dims, Ls, 1, 15)
    lat = Lattice(dims, Ls, prec=dw.DW_F64)
    lat.load_gauge(U)
    x = lat.pack(psi)
    y, ref = lat.empty().zero_(), lat.empty().zero_()

    def noalloc():
        mf = (ctypes.c_double * 1)(0.05)
        rc = dw.load_library().dw_apply_DdagD_noalloc(
            lat.handle, y.data_ptr(), x.data_ptr(), mf, 1,
            torch.cuda.current_stream().cuda_stream)
        assert rc == dw.DW_OK, dw.dw_last_error()

    assert launches(noalloc, "phi_kernel") == 1
    lat.DdagD(ref, x, 0.05)
    assert torch.equal(y, ref)
    lat.close()
