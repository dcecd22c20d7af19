"""What this library's speed is measured on: the calls a user makes, over the sizes they are made at.

A case names one public call (``op``), a lattice, boundary conditions, a precision, a number of
right-hand sides and, where it matters, a polynomial, a small space and field phases.  Inputs are
synthetic: random SU(3) links exp(i 0.2 H) near the free field, Gaussian spinors, spin-colour point
sources for the solves, and random orthonormal vectors with random signs as small-space banks of the
operator calls (their arithmetic does not depend on the vectors being eigenvectors).
"""
import math

import numpy as np
import torch

import paper_1111_6288_gb300 as ovl

M0 = -1.5
HW_NORM = 6.5  # |4 + m0| + 4, the bound the library uses by default
LINK_EPS = 0.2
PREC = {"f64": ovl.OV_PREC_F64, "f32": ovl.OV_PREC_F32, "f16": ovl.OV_PREC_F16, "bf16": ovl.OV_PREC_BF16}
BC = {"p": ovl.OV_BC_PERIODIC, "a": ovl.OV_BC_ANTIPERIODIC, "d": ovl.OV_BC_DIRICHLET}
BC_FACTOR = {"p": 1.0, "a": -1.0, "d": 0.0}
FIELD_STEP = (2.0 / 3.0) * 1e-4  # q E of the smallest background field


def _case(op, dims, **kw):
    c = dict(op=op, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], bc="pppa", prec="f32", nrhs=1, nphase=0, nev=0,
             degree=0, sqrt_eps=0.02, mass=0.0, tol=0.0)
    c.update(kw)
    return c


def listed():
    named = {
        # one Wilson application on the smallest lattice: what a call costs when the GPU has nothing to do
        "wilson-4x4-f64": _case("wilson", (4, 4, 4, 4), prec="f64"),
        # D_w on the 12 columns of a propagator in a background field (residual checks, contractions)
        "wilson-24x48-f32-12": _case("wilson", (24, 24, 24, 48), bc="dppd", nrhs=12, nphase=1),
        # the plain method on its smallest configuration: degree 200, 8 exact modes, FP64
        "sign-4x4-f64": _case("sign", (4, 4, 4, 4), prec="f64", nev=8, degree=200, sqrt_eps=math.sqrt(0.002)),
        # D(m) as the solver's inner loop applies it: one source, the full degree, 50 exact modes
        "overlap-16x32-f32": _case("overlap", (16, 16, 16, 32), nev=50, degree=527, mass=0.02),
        # the same in FP64: the true residual of every solve
        "overlap-16x32-f64": _case("overlap", (16, 16, 16, 32), prec="f64", nev=50, degree=527, mass=0.02),
        # a batch of 12 sources x 2 field values, at the degree of a late cycle of an adaptive solve
        "overlap-24x48-f32-24": _case("overlap", (24, 24, 24, 48), bc="dppd", nrhs=24, nphase=2, degree=120, mass=0.02),
        # 12 sources with 16-bit storage of links and recurrence vectors
        "overlap-16x32-f16-12": _case("overlap", (16, 16, 16, 32), prec="f16", nrhs=12, degree=120, mass=0.02),
        # extents that are multiples of nothing in particular, a few systems, a small space per field value
        "overlap-ragged-f32-5": _case("overlap", (10, 9, 14, 22), bc="dppd", nrhs=5, nphase=2, nev=12, degree=120,
                                      mass=0.05),
        # the exact small space of a batch: 24 chiral systems on a bank of 100
        "project-16x32-f32-24": _case("project", (16, 16, 16, 32), nrhs=24, nev=100),
        # a whole mixed-precision solve of the 12 sources of one propagator
        "solve-8x16-f32-12": _case("solve", (8, 8, 8, 16), nrhs=12, degree=210, sqrt_eps=0.05, mass=0.05, tol=1e-12),
        # the set-up of every configuration: low modes of Q
        "eigen-8x16-16": _case("eigen", (8, 8, 8, 16), prec="f64", nev=16, degree=64, sqrt_eps=0.05, tol=1e-8),
        # the field derivative of D(m) on 12 propagator columns
        "derivative-8x16-12": _case("derivative", (8, 8, 8, 16), bc="dppd", prec="f64", nrhs=12, nphase=1, degree=120,
                                    mass=0.02),
    }
    return [dict(c, name=n) for n, c in named.items()]


def _dims(rng, most):
    """Extents 3..24 (time 4..48), the site count spread over its logarithm between 200 and `most`."""
    want = math.exp(rng.uniform(math.log(200.0), math.log(float(most))))
    while True:
        d = [rng.randint(3, 24) for _ in range(3)] + [rng.randint(4, 48)]
        if 0.6 * want <= d[0] * d[1] * d[2] * d[3] <= min(want * 1.6, most):
            return d


def draw(rng):
    op = rng.choice(["wilson", "sign", "overlap", "overlap", "overlap", "project", "solve", "eigen", "derivative"])
    batch = rng.choice([1, 1, 2, 3, 5, 8, 12, 17, 24])
    field = rng.random() < 0.5
    nphase = rng.choice([1, 2]) if field and batch > 1 else int(field)
    bc = "dppd" if field else "pppa"
    if op == "wilson":
        prec = rng.choice(["f64", "f32", "f32", "f16", "bf16"])
        most = 7_900_000 // batch // (4 if prec == "f64" else 1)
        return _case(op, _dims(rng, min(most, 663552)), bc=bc, prec=prec, nrhs=batch, nphase=nphase)
    if op in ("sign", "overlap"):
        prec = rng.choice(["f64", "f32", "f32", "f32", "f16"])
        # the polynomial is evaluated below its interval on the few modes near zero that Dirichlet
        # faces bring, so its degree stays low there
        sqrt_eps = rng.choice([0.02, 0.05])
        degree = int(rng.uniform(1.2, 2.4 if field else 10.0) / sqrt_eps)
        most = {"f64": 60_000_000, "f32": 600_000_000, "f16": 200_000_000}[prec] // (batch * degree)
        d = _dims(rng, max(260, min(most, 300_000)))
        nev = rng.choice([0, 4, 12, 31, 50]) if d[0] * d[1] * d[2] * d[3] <= 132_000 else 0
        return _case(op, d, bc=bc, prec=prec, nrhs=batch, nphase=nphase, nev=nev, degree=degree, sqrt_eps=sqrt_eps,
                     mass=rng.choice([0.0, 0.02, 0.1]) if op == "overlap" else 0.0)
    if op == "project":
        nev = rng.choice([3, 16, 31, 50, 64, 100])
        return _case(op, _dims(rng, 13_000_000 // nev if nev > 99 else 131_072), nrhs=batch, nev=nev,
                     prec=rng.choice(["f32", "f32", "f64"]))
    if op == "solve":
        batch = rng.choice([1, 2, 6, 12])
        return _case(op, _dims(rng, 90_000 // batch), nrhs=batch, degree=210, sqrt_eps=0.05,
                     mass=rng.choice([0.05, 0.1]), tol=1e-12)
    if op == "eigen":
        return _case(op, _dims(rng, 6000), prec="f64", nev=rng.choice([4, 8, 12, 16]), degree=64, sqrt_eps=0.05, tol=1e-8)
    return _case(op, _dims(rng, 90_000 // batch), bc="dppd", prec="f64", nrhs=batch, nphase=max(nphase, 1),
                 degree=rng.randint(40, 120), mass=0.02)


# ---- inputs -------------------------------------------------------------------------------------


def _volume(c):
    return c["lx"] * c["ly"] * c["lz"] * c["lt"]


def _sites(c):
    return (c["lt"], c["lz"], c["ly"], c["lx"])


def _randn(gen, shape):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=gen, dtype=torch.float64, device="cuda"))


def _mm(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _links(c, gen):
    """U[4, t, z, y, x, 3, 3] = exp(i LINK_EPS H), H Hermitian and traceless with Gaussian coefficients."""
    g = torch.randn((4,) + _sites(c) + (8,), generator=gen, dtype=torch.float64, device="cuda")
    h = torch.zeros((4,) + _sites(c) + (3, 3), dtype=torch.complex128, device="cuda")
    for (i, j), k in (((0, 1), 0), ((0, 2), 3), ((1, 2), 5)):
        z = torch.complex(g[..., k], -g[..., k + 1])
        h[..., i, j], h[..., j, i] = z, z.conj()
    d3, d8 = g[..., 2], g[..., 7] / math.sqrt(3.0)
    h[..., 0, 0], h[..., 1, 1], h[..., 2, 2] = d3 + d8, d8 - d3, -2.0 * d8
    h *= 1j * LINK_EPS / 8  # exp(a) = exp(a / 8)^8; the series of exp(a / 8) ends below 1e-17
    out = torch.eye(3, dtype=torch.complex128, device="cuda").expand_as(h).clone()
    for k in range(12, 0, -1):
        out = _mm(h, out) / k
        for i in range(3):
            out[..., i, i] += 1.0
    for _ in range(3):
        out = _mm(out, out)
    return out.contiguous()


def _spinors(c, gen, n):
    x = torch.empty((n,) + _sites(c) + (4, 3), dtype=torch.complex128 if c["prec"] == "f64" else torch.complex64,
                    device="cuda")
    for j in range(n):
        v = _randn(gen, x.shape[1:])
        x[j] = v / torch.linalg.vector_norm(v)
    return x


def _phases(c):
    """One field phase per right-hand side, the right-hand sides of a phase together (None: no field)."""
    if c["nphase"] == 0:
        return None
    return [FIELD_STEP * (1 + j * c["nphase"] // c["nrhs"]) for j in range(c["nrhs"])]


def _banks(c, gen):
    """(phase, vectors, eigenvalues) of the small space of every field phase of the case."""
    for p in sorted(set(_phases(c) or [0.0])):
        v = torch.empty((c["nev"],) + _sites(c) + (4, 3), dtype=torch.complex64, device="cuda")
        for j in range(c["nev"]):
            v[j] = _randn(gen, v.shape[1:])
        lam = 0.01 * torch.randn(c["nev"], generator=gen, dtype=torch.float64, device="cuda").cpu().numpy()
        yield p, v, lam


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    U = _links(case, gen)
    if case["op"] == "solve":  # spin-colour point sources at one site
        n = torch.randint(_volume(case), (1,), generator=gen, device="cuda").item()
        x = torch.zeros((case["nrhs"], _volume(case), 12), dtype=torch.complex128, device="cuda")
        for j in range(case["nrhs"]):
            x[j, n, j % 12] = 1.0
        x = x.view((case["nrhs"],) + _sites(case) + (4, 3))
    elif case["op"] == "eigen":
        x = None
    else:
        x = _spinors(case, gen, case["nrhs"])
    return U, x, gen


def prepare(case, seed):
    U, x, gen = _inputs(case, seed)
    solve = case["op"] == "solve"
    ctx = ovl.Context(ovl.Params(
        dims=(case["lx"], case["ly"], case["lz"], case["lt"]), bc=[BC[b] for b in case["bc"]], m0=M0,
        eps=case["sqrt_eps"] ** 2, poly_degree=max(1, case["degree"]), poly_kind=1, precision=PREC[case["prec"]],
        inner_precision=ovl.OV_PREC_F32 if solve else ovl.OV_PREC_F64, max_nrhs=case["nrhs"],
        adaptive_order=int(solve)))
    ctx.set_gauge(U)
    if case["op"] in ("sign", "overlap", "project", "derivative"):
        for p, v, lam in _banks(case, gen):
            if len(lam) or p:
                ovl.deflate(ctx, v, lam, phase=p)
    st = dict(case=case, ctx=ctx, x=x, phase=_phases(case))
    if x is not None:
        st["out"] = torch.zeros_like(x)
        if case["op"] == "project":
            st["out2"] = torch.zeros_like(x)
    torch.cuda.synchronize()
    return st


def run(state):
    case, ctx, x, phase = state["case"], state["ctx"], state["x"], state["phase"]
    op = case["op"]
    if op == "wilson":
        return ovl.apply_wilson(ctx, x, state["out"], phase=phase)
    if op == "sign":
        return ovl.apply_sign_Hw(ctx, x, state["out"], phase=phase)
    if op == "overlap":
        return ovl.apply_overlap(ctx, x, state["out"], mass=case["mass"], phase=phase)
    if op == "project":
        return ovl.project_small(ctx, x, state["out"], state["out2"])
    if op == "derivative":
        return ovl.apply_dDdphi(ctx, x, state["out"], case["mass"], phase=phase)
    if op == "solve":
        sol = state["out"].zero_()
        ovl.solve_overlap(ctx, x, sol, case["mass"], tol=case["tol"], phase=phase)
        return sol
    return ovl.eigensolve_Q(ctx, case["nev"], tol=case["tol"])[0]


def work(case):
    """Inputs once, outputs once; 1368 floating-point operations per site and Wilson application."""
    V, k, n, N = _volume(case), case["nrhs"], case["degree"], case["nev"]
    cplx = 16 if case["prec"] == "f64" else 8
    gauge, vec = 4 * 9 * V * 16, 12 * V * cplx
    banks = max(1, case["nphase"]) * N * vec
    op = case["op"]
    if op == "wilson":
        return {"bytes": gauge + 2 * k * vec, "flops": 1368.0 * V * k}
    if op == "project":
        return {"bytes": banks + 3 * k * vec, "flops": 3 * 8.0 * 12 * V * N * k}
    if op in ("sign", "overlap"):
        return {"bytes": gauge + banks + 2 * k * vec, "flops": ((2 * n + 1) * 1368.0 + 3 * 96.0 * N) * V * k}
    if op == "derivative":
        return {"bytes": gauge + 2 * k * vec, "flops": 4 * n * 1368.0 * V * k}
    if op == "solve":  # about 40 inner iterations on two chiral sectors, one sign application each
        return {"bytes": gauge + 2 * k * vec, "flops": 80 * 2 * n * 1368.0 * V * k}
    return {"bytes": gauge, "flops": 2 * N * 500 * 1368.0 * V}  # about 500 filter steps on a double-width block


# ---- the same in plain torch, FP64 ----------------------------------------------------------------

# gamma_mu = [[0, G], [G^+, 0]] in the chiral basis: row a of G has its entry in column col[a]
_G = (((1, 0), (-1j, -1j)), ((1, 0), (-1, 1)), ((0, 1), (-1j, 1j)), ((0, 1), (1, 1)))


def _apply_gamma(mu, h):
    col, val = _G[mu]
    out = torch.empty_like(h)
    for a in range(2):
        out[..., a, :] = val[a] * h[..., 2 + col[a], :]
        out[..., 2 + col[a], :] = complex(val[a]).conjugate() * h[..., a, :]
    return out


def _hops(U, x, c, phi, mu):
    """(1 - gamma) U x(n + mu) and (1 + gamma) U^+ x(n - mu), for one right-hand side [t, z, y, x, 4, 3]."""
    f = BC_FACTOR[c["bc"][mu]]
    ax = 3 - mu
    u = U[mu]
    if mu == 0 and phi:
        t = torch.arange(c["lt"], device="cuda", dtype=torch.float64)
        u = u * torch.polar(torch.ones_like(t), phi * t)[:, None, None, None, None, None]
    L = x.shape[ax]
    fwd = torch.roll(x, -1, ax)
    fwd.select(ax, L - 1).mul_(f)
    fwd = (u[..., None, :, :] * fwd[..., :, None, :]).sum(-1)
    bwd = (u.conj()[..., None, :, :] * x[..., :, :, None]).sum(-2)
    bwd = torch.roll(bwd, 1, ax)
    bwd.select(ax, 0).mul_(f)
    return fwd - _apply_gamma(mu, fwd), bwd + _apply_gamma(mu, bwd)


def _g5(x):
    y = x.clone()
    y[..., 2:, :].neg_()
    return y


def _hw(U, x, c, phi):
    out = (4.0 + M0) * x
    for mu in range(4):
        f, b = _hops(U, x, c, phi, mu)
        out -= 0.5 * f
        out -= 0.5 * b
    return _g5(out)


def _dhw(U, x, c, phi):
    """d H_w / d phi: the x hops with their phases differentiated."""
    f, b = _hops(U, x, c, phi, 0)
    t = torch.arange(c["lt"], device="cuda", dtype=torch.float64)[:, None, None, None, None, None]
    return _g5(-0.5j * t * (f - b))


def _coeffs(c):
    return ovl.minimax_coeffs(c["degree"], c["sqrt_eps"] ** 2)[0]


def _poly(U, x, c, phi, cf):
    """Q P(Q^2) x by the forward recurrence of the T_k."""
    eps = c["sqrt_eps"] ** 2

    def y(v):
        return (2.0 / HW_NORM**2 * _hw(U, _hw(U, v, c, phi), c, phi) - (1.0 + eps) * v) / (1.0 - eps)

    a, b = x, y(x)
    s = cf[0] * a + cf[1] * b
    for k in range(2, len(cf)):
        a, b = b, 2.0 * y(b) - a
        s += cf[k] * b
    return _hw(U, s, c, phi) / HW_NORM


def _dpoly(U, x, c, phi, cf):
    """The phi-derivative of Q P(Q^2) x with x fixed."""
    eps = c["sqrt_eps"] ** 2
    s2 = 2.0 / HW_NORM**2 / (1.0 - eps)

    def y(v, dv):
        h, dh = _hw(U, v, c, phi), _dhw(U, v, c, phi) + _hw(U, dv, c, phi)
        return (s2 * _hw(U, h, c, phi) - (1.0 + eps) / (1.0 - eps) * v,
                s2 * (_dhw(U, h, c, phi) + _hw(U, dh, c, phi)) - (1.0 + eps) / (1.0 - eps) * dv)

    a, da = x, torch.zeros_like(x)
    b, db = y(a, da)
    s, ds = cf[0] * a + cf[1] * b, cf[1] * db
    for k in range(2, len(cf)):
        nb, ndb = y(b, db)
        a, da, b, db = b, db, 2.0 * nb - a, 2.0 * ndb - da
        s, ds = s + cf[k] * b, ds + cf[k] * db
    return (_dhw(U, s, c, phi) + _hw(U, ds, c, phi)) / HW_NORM


def _project(bank, x):
    """(V diag(s) V^+ x, x - V V^+ x) with V the vectors orthonormalised in order."""
    if bank is None:
        return torch.zeros_like(x), x
    v, sg = bank
    cc = v.conj() @ x.reshape(-1)
    return (v.T @ (sg * cc)).view(x.shape), x - (v.T @ cc).view(x.shape)


def _cost(c):
    """Seconds the plain evaluation takes, roughly."""
    n = {"wilson": 1, "sign": 2 * c["degree"], "overlap": 2 * c["degree"], "derivative": 7 * c["degree"]}.get(c["op"], 0)
    return c["nrhs"] * n * (1e-3 + 2e-8 * _volume(c))


def exact(case, seed):
    c = dict(case)
    if c["op"] == "solve" or (c["op"] == "eigen" and _volume(c) > 260) or _cost(c) > 18.0:
        return None
    U, x, gen = _inputs(c, seed)
    if c["op"] == "eigen":
        n = 12 * _volume(c)
        h = torch.empty((n, n), dtype=torch.complex128, device="cuda")
        for j in range(n):
            e = torch.zeros(n, dtype=torch.complex128, device="cuda")
            e[j] = 1.0
            h[:, j] = _hw(U, e.view(_sites(c) + (4, 3)), c, 0.0).reshape(-1)
        w = np.linalg.eigvalsh(h.cpu().numpy()) / HW_NORM
        return w[np.argsort(np.abs(w), kind="stable")][: c["nev"]]
    phase = _phases(c) or [0.0] * c["nrhs"]
    banks = {}
    if c["op"] in ("sign", "overlap", "project") and c["nev"]:
        for p, v, lam in _banks(c, gen):
            v = v.view(c["nev"], -1).to(torch.complex128)
            for _ in range(2):
                low = torch.linalg.cholesky(v.conj() @ v.T)  # <v_i, v_j> = L L^+: conj(L^{-1}) v is orthonormal
                v = torch.linalg.inv(low).conj() @ v
            banks[p] = (v, torch.as_tensor(np.where(lam >= 0, 1.0, -1.0), device="cuda").to(torch.complex128))
    cf = _coeffs(c) if c["op"] in ("sign", "overlap", "derivative") else None
    outs = []
    for j in range(c["nrhs"]):
        xj, phi = x[j].to(torch.complex128), phase[j]
        if c["op"] == "wilson":
            outs.append(_g5(_hw(U, xj, c, phi)))
            continue
        if c["op"] == "derivative":
            outs.append((1.0 - 0.5 * c["mass"]) * _g5(_dpoly(U, xj, c, phi, cf)))
            continue
        ys, xp = _project(banks.get(phi), xj)
        if c["op"] == "project":
            outs.append((ys, xp))
            continue
        sign = ys + _poly(U, xp, c, phi, cf)
        m = c["mass"]
        outs.append(sign if c["op"] == "sign" else (1.0 - 0.5 * m) * (xj + _g5(sign)) + m * xj)
    if c["op"] == "project":
        return torch.stack([o[0] for o in outs]), torch.stack([o[1] for o in outs])
    return torch.stack(outs)
