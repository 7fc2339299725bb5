"""Performance cases of the domain-wall library: the calls its users make, from
one apply on a 4^4 test lattice to the Dhop of the 32^3 x 64 x 12 benchmark.

``listed()`` names the fixed cases, ``draw(rng)`` gives further ones of the same
ranges, ``prepare`` builds what a program holds before the call (the lattice
with its gauge field, packed source fields on the GPU), ``run`` is one call (or
the short fixed sequence of calls such a program makes), ``work`` its algorithmic
bytes and flops, ``tolerance`` how far two correct implementations may be apart
and ``exact`` the same result from plain torch in complex128.

A case is a dict of plain values:
  kind   "apply" (dw_apply_*), "schur" (dw_apply_schur and its adjoint), "solve"
         (dw_cg_solve / dw_solve_eo), "fields" (gauge load, pack, Dhop, unpack of a
         new configuration) or "host" (dw_apply_host)
  op     the operator ("dhop", "dhop_dag", "D", "Ddag", "DdagD"), for a solve "cg" or "eo"
  prec   storage precision of the fields (for a solve: of its inner iteration)
  Lx, Ly, Lz, Lt, Ls, nrhs, form ("mobius" / "shamir"), mf
  tune   the program tuned its launch tiles first (Lattice.tune, once per
         lattice shape; later lattices of the shape take the saved tile)
"""

import numpy as np
import torch

from paper_2112_01852_gb300 import dw
from paper_2112_01852_gb300.lattice import Lattice

M5 = 1.8
BC = (1, 1, 1, -1)
PREC = {"f64": dw.DW_F64, "f32": dw.DW_F32, "f16": dw.DW_F16}
DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}
REAL_BYTES = {"f64": 8, "f32": 4, "f16": 2}
OPS = {"dhop": dw.DW_OP_DHOP, "dhop_dag": dw.DW_OP_DHOP_DAG, "D": dw.DW_OP_D,
       "Ddag": dw.DW_OP_DDAG, "DdagD": dw.DW_OP_DDAGD}
# inner iterations of the solves, nominal (as at the listed sizes), for work()
SOLVE_ITERS = {"cg": 480, "eo": 290}
SOLVE_TOL = 1e-10


def _case(name, kind, op, prec, dims, Ls, nrhs=1, form="mobius", mf=0.01, tune=False):
    c = dict(name=name, kind=kind, op=op, prec=prec, Lx=dims[0], Ly=dims[1], Lz=dims[2],
             Lt=dims[3], Ls=Ls, nrhs=nrhs, form=form, mf=mf, tune=tune)
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # the smallest call: one hop on a unit-test lattice, launch latency
        _case("dhop_f32_4x4x4x4_ls8", "apply", "dhop", "f32", (4, 4, 4, 4), 8),
        # the benchmark: the Domain Wall kernel on the production lattice, tuned
        _case("dhop_f32_32x32x32x64_ls12", "apply", "dhop", "f32", (32, 32, 32, 64), 12,
              tune=True),
        # the normal operator of a 24^4 Moebius solve, tuned (light-quark mass)
        _case("ddagd_f32_24x24x24x24_ls16", "apply", "DdagD", "f32", (24, 24, 24, 24), 16,
              tune=True),
        # FP64 operator: true residuals, measurements in full precision
        _case("d_f64_16x16x16x16_ls16", "apply", "D", "f64", (16, 16, 16, 16), 16),
        # half-precision storage on the paper's 24^3 x 48 x 8 volume
        _case("dhop_dag_f16_24x24x24x48_ls8", "apply", "dhop_dag", "f16", (24, 24, 24, 48), 8),
        # a propagator's 12 spin-colour sources at once
        _case("ddagd_f32_16x16x16x32_ls12_12rhs", "apply", "DdagD", "f32", (16, 16, 16, 32), 12,
              nrhs=12),
        # odd extents and an odd Ls, Shamir form: nothing divides a warp or a tile
        _case("ddag_f32_11x10x7x18_ls9", "apply", "Ddag", "f32", (11, 10, 7, 18), 9,
              form="shamir", mf=0.02),
        # the even-odd operator and its adjoint, what each step of a preconditioned solve applies
        _case("schur_f32_24x24x24x24_ls16", "schur", "schur", "f32", (24, 24, 24, 24), 16),
        # a whole preconditioned mixed-precision solve of D x = eta
        _case("solve_eo_f32_16x16x16x32_ls12", "solve", "eo", "f32", (16, 16, 16, 32), 12,
              mf=0.05),
        # a whole mixed-precision CG on a small lattice, FP16 inner fields
        _case("solve_cg_f16_8x8x8x16_ls8", "solve", "cg", "f16", (8, 8, 8, 16), 8, mf=0.05),
        # a new configuration and source arrive: gauge load, pack, one hop, unpack
        _case("fields_f32_24x24x24x48_ls8", "fields", "dhop", "f32", (24, 24, 24, 48), 8),
        # fields that live in host memory: copies and operator in one call
        _case("host_d_f32_16x16x16x32_ls12", "host", "D", "f32", (16, 16, 16, 32), 12),
    ]


def _loguniform(rng, lo, hi):
    return float(np.exp(rng.uniform(np.log(lo), np.log(hi))))


def _dims(rng, v4, even):
    """Four extents with a volume near v4, x and t longest on average."""
    side = v4 ** 0.25
    while True:
        d = [side * _loguniform(rng, 0.6, 1.7) for _ in range(3)]
        d = [max(2, int(round(x / 2)) * 2 if even or rng.random() < 0.7 else int(round(x)))
             for x in d]
        d[0] = min(d[0], 48)
        t = v4 / (d[0] * d[1] * d[2])
        t = max(2, int(round(t / 2)) * 2 if even or rng.random() < 0.7 else int(round(t)))
        if t <= 96 and 0.5 * v4 <= d[0] * d[1] * d[2] * t <= 2.0 * v4:
            return (d[0], d[1], d[2], t)


def draw(rng):
    kind = rng.choices(["apply", "schur", "solve", "fields", "host"], [55, 15, 10, 10, 10])[0]
    form = "mobius" if rng.random() < 0.75 else "shamir"
    mf = rng.choice([0.005, 0.01, 0.02, 0.05])
    prec = rng.choices(["f32", "f64", "f16"], [60, 20, 20])[0]
    Ls = rng.choice([4, 5, 6, 7, 8, 9, 10, 12, 12, 16, 16])
    if kind == "solve":
        op = rng.choice(["cg", "eo"])
        dims = _dims(rng, _loguniform(rng, 1 << 9, 1 << 15), even=True)
        return _case(None, kind, op, rng.choice(["f32", "f16"]), dims, rng.choice([6, 8, 12]),
                     form=form, mf=0.05)
    # 4D sites: from a test lattice to the benchmark's 2^21; FP64 is bounded by
    # its arithmetic and is used on smaller lattices
    top = {"apply": 1 << 21, "schur": 1 << 20, "fields": 1 << 20, "host": 1 << 18}[kind]
    if prec == "f64":
        top = min(top, 1 << 18)
    v4 = _loguniform(rng, 1 << 8, top / 2.1)
    dims = _dims(rng, v4, even=kind == "schur")
    if kind == "schur":
        return _case(None, kind, "schur", prec, dims, Ls, form=form, mf=mf)
    if kind == "fields":
        return _case(None, kind, "dhop", prec, dims, Ls, form=form, mf=mf)
    op = rng.choice(["dhop", "dhop_dag", "D", "Ddag", "DdagD"])
    if kind == "host":
        return _case(None, kind, op, prec, dims, Ls, form=form, mf=mf)
    nrhs = rng.choice([1, 1, 1, 1, 2, 3, 12])
    sites = dims[0] * dims[1] * dims[2] * dims[3] * Ls
    while nrhs > 1 and nrhs * sites > 8_000_000:
        nrhs -= 1
    return _case(None, kind, op, prec, dims, Ls, nrhs=nrhs, form=form, mf=mf,
                 tune=nrhs == 1 and sites < 3_000_000 and rng.random() < 0.3)


# ---------------------------------------------------------------------------
# inputs, on the GPU and from the seed alone

def _shape(case):
    dims = (case["Lx"], case["Ly"], case["Lz"], case["Lt"])
    return dims, dims[0] * dims[1] * dims[2] * dims[3], case["Ls"], case["nrhs"]


def _bc(case):
    return (1.5, 0.5) if case["form"] == "mobius" else (1.0, 0.0)


def _links(case, seed):
    """Near-unit SU(3) links: the first two rows of 1 + 0.3 i H, H Hermitian Gaussian,
    orthonormalised, the third their cross product; complex128 (V4, 4, 3, 3)."""
    _, V4, _, _ = _shape(case)
    g = torch.Generator(device="cuda").manual_seed(2 * seed + 1)
    a = torch.randn(V4 * 4, 3, 3, 2, generator=g, device="cuda", dtype=torch.float64)
    a = torch.view_as_complex(a)
    a = 0.15j * (a + a.transpose(1, 2).conj())
    a += torch.eye(3, device="cuda", dtype=torch.complex128)
    r0, r1 = a[:, 0], a[:, 1]
    r0 = r0 / torch.linalg.vector_norm(r0, dim=1, keepdim=True)
    r1 = r1 - (r0.conj() * r1).sum(1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
    r2 = torch.linalg.cross(r0.conj(), r1.conj())
    return torch.stack([r0, r1, r2], 1).reshape(V4, 4, 3, 3)


def _source(case, seed):
    """Complex Gaussian spinors, canonical complex128 (nrhs, V4, Ls, 4, 3), with
    values that the storage precision holds exactly (a solve's right-hand side is FP64)."""
    _, V4, Ls, nrhs = _shape(case)
    g = torch.Generator(device="cuda").manual_seed(2 * seed + 2)
    dt = torch.float32 if case["prec"] != "f64" else torch.float64
    x = torch.randn(nrhs, V4, Ls, 4, 3, 2, generator=g, device="cuda", dtype=dt)
    if case["prec"] == "f16":
        x = x.half()
    return torch.view_as_complex(x.double())


_TILES = {}  # the tiles a program keeps once it has tuned a lattice shape


def _tune(lat, case):
    ops = {"DdagD": ["D", "Ddag"]}.get(case["op"], [case["op"]])
    for op in ops:
        key = (lat.dims, lat.Ls, lat.prec, op)
        if key not in _TILES:
            _TILES[key] = lat.tune(OPS[op], case["nrhs"])
        else:
            spt, tx, variant, zblk, sgrp = _TILES[key]
            lat.set_tile(OPS[op], spt, tx, variant, nrhs=case["nrhs"], zblk=zblk, sgrp=sgrp)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    dims, _, Ls, nrhs = _shape(case)
    b, c = _bc(case)
    kind = case["kind"]
    prec = dw.DW_F64 if kind == "solve" else PREC[case["prec"]]
    lat = Lattice(dims, Ls, kind=dw.DW_MOBIUS if case["form"] == "mobius" else dw.DW_SHAMIR,
                  M5=M5, b=b, c=c, prec=prec, bc=BC)
    links, src = _links(case, seed), _source(case, seed)
    dw.dw_load_gauge(lat.handle, links.data_ptr(), _stream())
    st = {"case": case, "lat": lat, "mf": [case["mf"]] * nrhs}
    if kind == "fields":
        st.update(links=links, src=src, x=lat.empty(nrhs).zero_(), y=lat.empty(nrhs).zero_(),
                  dst=torch.empty_like(src))
        torch.cuda.synchronize()
        return st
    x = lat.empty(nrhs).zero_()
    dw.dw_pack_fermion(lat.handle, x.data_ptr(), prec, src.data_ptr(), nrhs, _stream())
    if case["tune"]:
        _tune(lat, case)
    if kind == "apply":
        st.update(x=x, y=lat.empty(nrhs).zero_())
    elif kind == "schur":
        even, odd = lat.empty_eo(nrhs).zero_(), lat.empty_eo(nrhs).zero_()
        dw.dw_eo_split(lat.handle, even.data_ptr(), odd.data_ptr(), x.data_ptr(), prec, nrhs,
                       _stream())
        st.update(x=odd, y=lat.empty_eo(nrhs).zero_(), z=lat.empty_eo(nrhs).zero_())
    elif kind == "solve":
        # a program solves for many sources: its first solve has set the solver up
        st.update(b=x, x=lat.empty(nrhs).zero_())
        _solve(st, maxit=2)
    else:  # host: pinned host buffers, as a program that streams fields keeps them
        xin = torch.empty(x.numel(), dtype=torch.uint8, pin_memory=True)
        xin.copy_(x)
        yout = torch.empty(x.numel(), dtype=torch.uint8, pin_memory=True)
        yout.zero_()
        st.update(x=xin, y=yout)
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------
# the calls

def _solve(st, maxit):
    case, lat = st["case"], st["lat"]
    st["x"].zero_()
    solve = lat.cg if case["op"] == "cg" else lat.solve_eo
    return solve(st["x"], st["b"], st["mf"], case["nrhs"], tol=SOLVE_TOL, maxit=maxit,
                 mode=PREC[case["prec"]])


def _apply(lat, op, y, x, mf, nrhs):
    if op == "dhop" or op == "dhop_dag":
        lat.dhop(y, x, nrhs, dag=op == "dhop_dag")
    elif op == "D":
        lat.D(y, x, mf, nrhs)
    elif op == "Ddag":
        lat.Ddag(y, x, mf, nrhs)
    else:
        lat.DdagD(y, x, mf, nrhs)


def run(st):
    case, lat = st["case"], st["lat"]
    kind, nrhs = case["kind"], case["nrhs"]
    dt = DTYPE[case["prec"]]
    if kind == "apply":
        _apply(lat, case["op"], st["y"], st["x"], st["mf"], nrhs)
        return st["y"].view(dt)
    if kind == "schur":
        h, s = lat.handle, _stream()
        dw.dw_apply_schur(h, st["y"].data_ptr(), st["x"].data_ptr(), st["mf"], nrhs, 0, s)
        dw.dw_apply_schur(h, st["z"].data_ptr(), st["y"].data_ptr(), st["mf"], nrhs, 1, s)
        return [st["y"].view(dt), st["z"].view(dt)]
    if kind == "solve":
        _solve(st, maxit=5000)
        return st["x"].view(torch.float64)
    if kind == "fields":
        s = _stream()
        dw.dw_load_gauge(lat.handle, st["links"].data_ptr(), s)
        dw.dw_pack_fermion(lat.handle, st["x"].data_ptr(), lat.prec, st["src"].data_ptr(), nrhs, s)
        lat.dhop(st["y"], st["x"], nrhs)
        dw.dw_unpack_fermion(lat.handle, st["dst"].data_ptr(), st["y"].data_ptr(), lat.prec, nrhs,
                             s)
        return {"packed": st["x"].view(dt), "dhop": torch.view_as_real(st["dst"])}
    mf = st["mf"] if case["op"] in ("D", "Ddag", "DdagD") else None
    lat.apply_host(OPS[case["op"]], st["y"], st["x"], mf, nrhs)
    return st["y"].view(dt)


def work(case):
    """Each input once, each output once, the links once; 1320 flop per hop of a 5D
    site, 192 (Moebius) or 96 (Shamir) for the fifth-dimension terms of D."""
    _, V4, Ls, nrhs = _shape(case)
    rb = REAL_BYTES[case["prec"]]
    sites = V4 * Ls * nrhs
    local = 192 if case["form"] == "mobius" else 96
    field, links = 24 * rb * sites, 72 * rb * V4
    kind, op = case["kind"], case["op"]
    if kind == "schur":  # in and two results, half-volume fields; two hops each, A and A^-1
        return {"bytes": 3 * field / 2 + links, "flops": 2 * sites * (1320 + local + 96)}
    if kind == "solve":
        hops = {"cg": 2 * (1320 + local) + 6 * 24, "eo": 2 * (1320 + local + 96) + 3 * 24}[op]
        n = SOLVE_ITERS[op]
        per_iter = {"cg": 7, "eo": 3.5}[op] * field + 2 * links
        return {"bytes": n * per_iter, "flops": n * sites * hops}
    if kind == "fields":  # complex128 links and source in, packed field and complex128 result out
        return {"bytes": 72 * 8 * V4 + 2 * 24 * 8 * sites + field, "flops": 1320 * sites}
    per = {"dhop": 1320, "dhop_dag": 1320, "D": 1320 + local, "Ddag": 1320 + local,
           "DdagD": 2 * (1320 + local)}[op]
    return {"bytes": 2 * field + links, "flops": per * sites}


def tolerance(case):
    """About four times what was measured between two orders of the hop sum (one apply:
    8e-8 at FP32, 6e-6 at FP16) and, for the solves, between reliable-update thresholds
    (2e-9; both sides stop at a residual of 1e-10).  FP16 operators that pass through an
    intermediate FP16 field may round that field elsewhere (2^-11 per value)."""
    kind, prec = case["kind"], case["prec"]
    if kind == "solve":
        return {"rel": 2e-8, "max": 4e-7}
    if prec == "f64":
        return {"rel": 1e-15, "max": 1e-14}
    if prec == "f32":
        return {"rel": 4e-7, "max": 4e-6}
    if kind == "schur" or case["op"] == "DdagD":
        return {"rel": 1e-3, "max": 1e-2}
    return {"rel": 1e-4, "max": 4e-3}


# ---------------------------------------------------------------------------
# the same results from plain torch, complex128
#   gamma_k = [[0, i s_k], [-i s_k, 0]], gamma_4 = [[0, 1], [1, 0]], P+ the upper spins

def _gammas():
    s = [np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]]),
         np.array([[1, 0], [0, -1]], complex)]
    z = np.zeros((2, 2))
    g = [np.block([[z, 1j * m], [-1j * m, z]]) for m in s]
    return g + [np.block([[z, np.eye(2)], [np.eye(2), z]])]


def _spin(m, psi):
    """4 x 4 matrix with one entry per row on the spin index (axis -2)."""
    rows = []
    for i in range(4):
        j = int(np.argmax(np.abs(m[i])))
        rows.append(complex(m[i, j]) * psi[..., j, :])
    return torch.stack(rows, -2)


def _colour(U, psi):
    """U (sites, 3, 3) on the last axis of psi (nrhs, sites, Ls, 4, 3)."""
    out = torch.zeros_like(psi)
    for a in range(3):
        for k in range(3):
            out[..., a] += U[None, :, None, None, a, k] * psi[..., k]
    return out


def _hop(psi, U, case, dag):
    dims, V4, Ls, _ = _shape(case)
    x = torch.arange(V4, device=psi.device)
    out = torch.zeros_like(psi)
    stride = 1
    for mu, g in enumerate(_gammas()):
        L = dims[mu]
        pos = (x // stride) % L
        up = torch.where(pos == L - 1, x - (L - 1) * stride, x + stride)
        sign = 1.0 if dag else -1.0
        f = torch.where(pos == L - 1, float(BC[mu]), 1.0).to(U.dtype)[:, None, None]
        Um = U[:, mu] * f
        v = _colour(Um, psi[:, up])
        out += v
        out += sign * _spin(g, v)
        v = _colour(Um.transpose(1, 2).conj(), psi)  # at x, belongs to x + mu
        v = v - sign * _spin(g, v)
        out[:, up] += v
        del v
        stride *= L
    return out


def _K(psi, mf, dag):
    """K psi along s (axis 2); the adjoint has the chiralities exchanged."""
    dn, up = torch.roll(psi, 1, 2), torch.roll(psi, -1, 2)  # slices s-1, s+1
    dn[:, :, 0] *= -mf
    up[:, :, -1] *= -mf
    if dag:
        dn, up = up, dn
    return torch.cat([dn[..., :2, :], up[..., 2:, :]], -2)


def _D(psi, U, case, dag):
    b, c = _bc(case)
    mf = case["mf"]
    if not dag:
        phi = b * psi + c * _K(psi, mf, False)
        return (4 - M5) * phi - 0.5 * _hop(phi, U, case, False) + psi - _K(psi, mf, False)
    w = (4 - M5) * psi - 0.5 * _hop(psi, U, case, True)
    return b * w + c * _K(w, mf, True) + psi - _K(psi, mf, True)


def _local(psi, case, dag, inverse):
    """A = alpha + beta K (or its adjoint) or its inverse, as Ls x Ls matrices."""
    b, c = _bc(case)
    Ls = case["Ls"]
    alpha, beta = b * (4 - M5) + 1, c * (4 - M5) - 1
    lower = np.diag(np.ones(Ls - 1), -1)  # slice s from s-1
    lower[0, -1] += -case["mf"]
    m = {}
    for half, k in (("up", lower), ("lo", lower.T.copy())):
        a = alpha * np.eye(Ls) + beta * (k.T if dag else k)
        a = np.linalg.inv(a) if inverse else a
        m[half] = torch.tensor(a, device=psi.device, dtype=psi.dtype)
    return torch.cat([torch.einsum("ij,rxjsc->rxisc", m["up"], psi[..., :2, :]),
                      torch.einsum("ij,rxjsc->rxisc", m["lo"], psi[..., 2:, :])], -2)


def _H(psi, U, case, dag):
    b, c = _bc(case)
    if not dag:
        return -0.5 * _hop(b * psi + c * _K(psi, case["mf"], False), U, case, False)
    w = -0.5 * _hop(psi, U, case, True)
    return b * w + c * _K(w, case["mf"], True)


def _parity(case):
    (Lx, Ly, Lz, _), V4, _, _ = _shape(case)
    x = torch.arange(V4, device="cuda")
    return (x % Lx + x // Lx % Ly + x // (Lx * Ly) % Lz + x // (Lx * Ly * Lz)) % 2


def _schur(odd, U, case, dag):
    """Dhat (or its adjoint) of a full-lattice field that is zero on even sites."""
    p = _parity(case)[None, :, None, None, None]
    e = _local(_H(odd, U, case, dag) * (p == 0), case, dag, True)
    return (_local(odd, case, dag, False) - _H(e, U, case, dag)) * (p == 1)


def _internal(psi, prec):
    """Canonical (nrhs, sites, Ls, 4, 3) in the library's blocked layout, FP64 reals."""
    n, V, Ls = psi.shape[:3]
    r = torch.view_as_real(psi).reshape(n, V, Ls, 2, 2, 3, 2)  # half, spin, colour, re/im
    r = r.permute(0, 1, 2, 3, 5, 6, 4).reshape(n, V, Ls, 24)
    pad = -V % 32
    if pad:
        r = torch.cat([r, r.new_zeros(n, pad, Ls, 24)], 1)
    R = 2 if prec == "f64" else 4
    r = r.reshape(n, -1, 32, Ls, 24 // R, R).permute(0, 1, 3, 4, 2, 5)
    return r.reshape(-1)


def exact(case, seed):
    if case["kind"] == "solve":
        return None
    U, psi = _links(case, seed), _source(case, seed)
    prec, op = case["prec"], case["op"]
    if case["kind"] == "schur":
        p = _parity(case)
        y = _schur(psi * (p == 1)[None, :, None, None, None], U, case, False)
        z = _schur(y, U, case, True)
        odd = p == 1
        return [_internal(y[:, odd].contiguous(), prec), _internal(z[:, odd].contiguous(), prec)]
    if case["kind"] == "fields":
        return {"packed": _internal(psi, prec),
                "dhop": torch.view_as_real(_hop(psi, U, case, False))}
    if op in ("dhop", "dhop_dag"):
        y = _hop(psi, U, case, op == "dhop_dag")
    elif op in ("D", "Ddag"):
        y = _D(psi, U, case, op == "Ddag")
    else:
        y = _D(_D(psi, U, case, False), U, case, True)
    y = _internal(y, prec)
    return y.cpu() if case["kind"] == "host" else y
