"""The workloads whose speed this repository is measured by.

Each case is a call, or a short fixed sequence of calls, that a program using
this library makes through its public Python entry points: the operator on one
and on several right-hand sides, in each storage precision, from device and
from host memory; the solvers; the batch of independent systems; the deflation
solver; and the way of a configuration and its sources into and out of the
library.  Nothing is tuned beforehand: the launches are those a program gets
that calls the entry points as they are.

Lattices are given as T, Lx, Ly, Lz.  Gauge fields are Gaussian fluctuations of
strength `eps` around the unit links, projected to SU(3); sources are Gaussian
fields, or the spin x colour columns of a point source for propagators.
"""
import math

import torch

import paper_1405_0700_gb300 as P
from paper_1405_0700_gb300 import plq

PREC = {"f64": P.F64, "f32": P.F32, "f16": P.F16, "df64": P.DF64}
REAL_BYTES = {"f64": 8, "f32": 4, "f16": 2, "df64": 8}
SITE_BYTES = {"f64": 192, "f32": 96, "f16": 52, "df64": 192}


def listed():
    return [
        # the smallest call: a preconditioned operator application on a test-sized lattice (latency)
        dict(name="schur_f32_8c8", kind="schur", T=8, Lx=8, Ly=8, Lz=8, prec="f32", links=18, dagger=False),
        # the full operator in double precision, as a program checks residuals with
        dict(name="wilson_f64_16c32", kind="wilson", T=32, Lx=16, Ly=16, Lz=16, prec="f64", links=18, mu=0.0),
        # one half-lattice application in single precision with full links: the benchmark's operator
        dict(name="hop_f32_32c64", kind="hop", T=64, Lx=32, Ly=32, Lz=32, prec="f32", links=18, nrhs=1, parity=0),
        # the preconditioned adjoint operator in half-precision storage: an inner solver of the user's own
        dict(name="schur_f16_24c48", kind="schur", T=48, Lx=24, Ly=24, Lz=24, prec="f16", links=12, dagger=True),
        # the operator on fields that live in host memory (the benchmark's end-to-end call)
        dict(name="hop_host_f32_32c64", kind="hop_host", T=64, Lx=32, Ly=32, Lz=32, prec="f32", links=18, nrhs=1,
             parity=0),
        # the operator on the 12 spin x colour columns of a propagator at the largest lattice of the benchmark
        dict(name="hop_f32_x12_48c96", kind="hop", T=96, Lx=48, Ly=48, Lz=48, prec="f32", links=12, nrhs=12, parity=0),
        # the mixed-precision CG solve of the benchmark
        dict(name="cg_f32_24c48", kind="solve", method="cg", T=48, Lx=24, Ly=24, Lz=24, inner="f32", links=12, nrhs=1,
             residual="f64", kappa=0.12, mu=0.0, eps=0.3, point=False),
        # a twisted-mass BiCGstab solve with half-precision inner iterations and float-float residuals on a
        # lattice whose extents are no powers of two
        dict(name="bicg_f16_tm_20x12x28x36", kind="solve", method="bicgstab", T=36, Lx=20, Ly=12, Lz=28, inner="f16",
             links=12, nrhs=1, residual="df64", kappa=0.118, mu=0.05, eps=0.3, point=False),
        # a propagator: the 12 columns of a point source solved together
        dict(name="cg_f32_x12_24c48", kind="solve", method="cg", T=48, Lx=24, Ly=24, Lz=24, inner="f32", links=12,
             nrhs=12, residual="f64", kappa=0.121, mu=0.0, eps=0.25, point=True),
        # many independent systems of uneven lattices in one call (an ensemble's small jobs)
        dict(name="batch_f32_16", kind="batch", systems=16, big=24, inner="f32", links=12),
        # a configuration and 12 sources come in, the links are used once, 12 solutions go out
        dict(name="load_f32_x12_24c48", kind="load", T=48, Lx=24, Ly=24, Lz=24, prec="f32", links=12, nrhs=12),
        # deflation: the first right-hand sides of an incremental EigCG run with the paper's nev and m
        dict(name="eigcg_16c32", kind="eigcg", T=32, Lx=16, Ly=16, Lz=16, nev=10, m=60, sources=3, kappa=0.122,
             eps=0.1),
    ]


def _lattice(rng, lo, hi):
    """Even extents, T up to 96 and the others up to 48, of about exp(uniform(log lo, log hi)) sites."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    best = None
    for _ in range(400):
        L = [2 * rng.randint(2, 48)] + [2 * rng.randint(2, 24) for _ in range(3)]
        off = abs(math.log(L[0] * L[1] * L[2] * L[3] / want))
        if L[0] * L[1] * L[2] * L[3] <= hi and (best is None or off < best[0]):
            best = (off, L)
        if off < 0.2 and best[1] == L:
            break
    L = best[1] if best else [8, 8, 8, 8]
    return dict(T=L[0], Lx=L[1], Ly=L[2], Lz=L[3])


def draw(rng):
    kind = rng.choice(["schur", "wilson", "hop", "hop_host", "hop_n", "hop_n", "solve", "solve", "solve_n", "batch",
                       "load", "eigcg"])
    if kind == "schur":
        return dict(kind=kind, prec=rng.choice(["f32", "f16", "f64"]), links=rng.choice([18, 12]),
                    dagger=rng.random() < 0.5, **_lattice(rng, 4096, 48**3 * 24))
    if kind == "wilson":
        return dict(kind=kind, prec=rng.choice(["f64", "f32"]), links=rng.choice([18, 12]),
                    mu=rng.choice([0.0, round(rng.uniform(0.01, 0.1), 4)]), **_lattice(rng, 4096, 48**3 * 24))
    if kind == "hop":
        prec = rng.choice(["f32", "f16", "df64"])
        return dict(kind=kind, prec=prec, links=18 if prec == "df64" else rng.choice([18, 12]), nrhs=1,
                    parity=rng.randint(0, 1), **_lattice(rng, 16384, 48**3 * 96))
    if kind == "hop_host":
        return dict(kind=kind, prec=rng.choice(["f32", "f16"]), links=rng.choice([18, 12]), nrhs=rng.choice([1, 3]),
                    parity=rng.randint(0, 1), **_lattice(rng, 16384, 32**3 * 32))
    if kind == "hop_n":
        return dict(kind="hop", prec=rng.choice(["f32", "f32", "f16"]), links=rng.choice([18, 12]),
                    nrhs=rng.randint(2, 12), parity=rng.randint(0, 1), **_lattice(rng, 4096, 32**3 * 64))
    if kind in ("solve", "solve_n"):
        nrhs = 1 if kind == "solve" else rng.randint(2, 12)
        method = rng.choice(["cg", "cg", "bicgstab"])
        inner = rng.choice(["f32", "f32", "f16"])
        return dict(kind="solve", method=method, inner=inner, links=12 if inner == "f16" else rng.choice([12, 18]),
                    nrhs=nrhs, residual=rng.choice(["f64", "df64"]), kappa=round(rng.uniform(0.112, 0.121), 4),
                    mu=rng.choice([0.0, 0.05]) if nrhs == 1 else 0.0, eps=round(rng.uniform(0.25, 0.3), 3),
                    point=nrhs > 1 and method == "cg", **_lattice(rng, 4096, (24**3 * 48 if nrhs == 1 else 16**3 * 64)))
    if kind == "batch":
        return dict(kind=kind, systems=rng.randint(2, 16), big=rng.choice([16, 20, 24]), inner=rng.choice(["f32", "f16"]),
                    links=12)
    if kind == "load":
        prec = rng.choice(["f32", "f16"])
        return dict(kind=kind, prec=prec, links=rng.choice([12, 18]), nrhs=rng.randint(1, 12),
                    **_lattice(rng, 8192, 24**3 * 48))
    return dict(kind="eigcg", nev=rng.choice([6, 8, 10]), m=rng.choice([40, 60]), sources=rng.randint(2, 3),
                kappa=round(rng.uniform(0.118, 0.122), 4), eps=0.1, **_lattice(rng, 8192, 16**3 * 32))


# ---------------------------------------------------------------- inputs


def _dims(case):
    return (case["T"], case["Lx"], case["Ly"], case["Lz"])


def _rng(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 64 + what) % (1 << 62))
    return g


def _links(dims, eps, g):
    """SU(3) links around 1, canonical layout: complex128 (T, Lz, Ly, Lx, 4, 3, 3)."""
    T, Lx, Ly, Lz = dims
    U = torch.empty((T, Lz, Ly, Lx, 4, 3, 3), dtype=torch.complex128, device="cuda")
    one = torch.eye(3, dtype=torch.complex128, device="cuda")
    for mu in range(4):
        A = torch.randn((T, Lz, Ly, Lx, 3, 3), dtype=torch.complex64, device="cuda", generator=g).to(torch.complex128)
        M = one + (1j * eps / math.sqrt(2.0)) * (A + A.transpose(-1, -2).conj())
        del A
        a, b = M[..., 0, :], M[..., 1, :]
        a = a / torch.sqrt((a.real**2 + a.imag**2).sum(-1, keepdim=True))
        b = b - (a.conj() * b).sum(-1, keepdim=True) * a
        b = b / torch.sqrt((b.real**2 + b.imag**2).sum(-1, keepdim=True))
        U[..., mu, 0, :] = a
        U[..., mu, 1, :] = b
        for c in range(3):
            d, e = (c + 1) % 3, (c + 2) % 3
            U[..., mu, 2, c] = (a[..., d] * b[..., e] - a[..., e] * b[..., d]).conj()
        del M, a, b
    return U


def _gauss(dims, n, g):
    """n Gaussian spinor fields, canonical layout: complex128 (n, T, Lz, Ly, Lx, 4, 3)."""
    T, Lx, Ly, Lz = dims
    return torch.randn((n, T, Lz, Ly, Lx, 4, 3), dtype=torch.complex64, device="cuda", generator=g).to(torch.complex128)


def _point(dims, n, seed):
    """The first n spin x colour columns of a point source at a site that the seed picks."""
    T, Lx, Ly, Lz = dims
    b = torch.zeros((n, T, Lz, Ly, Lx, 4, 3), dtype=torch.complex128, device="cuda")
    s = int(seed) * 2654435761
    at = (s % T, s // 7 % Lz, s // 11 % Ly, s // 13 % Lx)
    for r in range(n):
        b[(r, *at, r // 3, r % 3)] = 1.0
    return b


def _source(case, seed):
    if case["point"]:
        return _point(_dims(case), case["nrhs"], seed)
    return _gauss(_dims(case), case["nrhs"], _rng(seed, 1))


def _batch_systems(case, seed):
    """(dims, kappa, eps) of each system: lattices of three sizes in turn, kappas spread over their range."""
    big = case["big"]
    sizes = [(16, 8, 8, 8), (32, 16, 16, 16), (2 * big, big, big, big)]
    return [(sizes[k % 3], 0.110 + 0.014 * ((k * 37 + int(seed) * 11) % 97) / 97.0, 0.3) for k in range(case["systems"])]


def _pack(ctx, phi, prec, n):
    out = ctx.empty_full(PREC[prec], n)
    ctx.pack_spinor(out, torch.view_as_real(phi), PREC[prec], n)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ctxs, xs, bs, kappas = [], [], [], []
        for k, (dims, kappa, eps) in enumerate(_batch_systems(case, seed)):
            ctx = P.Context(dims)
            g = _rng(seed, 2 + k)
            U = torch.view_as_real(_links(dims, eps, g))
            ctx.gauge_upload(U, 18, P.F64)
            ctx.gauge_upload(U, case["links"], PREC[case["inner"]])
            bs.append(_pack(ctx, _gauss(dims, 1, g), "f64", 1))
            xs.append(ctx.empty_full(P.F64))
            ctxs.append(ctx)
            kappas.append(kappa)
        return dict(case=case, ctxs=ctxs, xs=xs, bs=bs, kappas=kappas)

    dims = _dims(case)
    ctx = P.Context(dims)
    s = dict(case=case, ctx=ctx)
    U = torch.view_as_real(_links(dims, case.get("eps", 0.3), _rng(seed, 0)))
    if kind in ("hop", "hop_host", "schur", "wilson"):
        prec, n = case["prec"], case.get("nrhs", 1)
        ctx.gauge_upload(U, case["links"], PREC[prec])
        del U
        phi = _gauss(dims, n, _rng(seed, 1))
        full = _pack(ctx, phi, prec, n)
        del phi
        if kind == "wilson" or prec == "df64":
            s.update(inp=full, out=torch.empty_like(full))
            if prec == "df64":
                s["values"] = torch.empty(ctx.volume * 24, dtype=torch.float64, device="cuda")
        elif kind == "schur":
            e, o = ctx.halves(full, PREC[prec])
            s.update(inp=e, tmp=torch.empty_like(e), out=torch.empty_like(e))
        else:
            inp = ctx.halves(full, PREC[prec], n)[1 - case["parity"]].clone()
            if kind == "hop":
                s.update(inp=inp, out=torch.empty_like(inp))
            else:
                s["inp"] = torch.empty(inp.numel(), dtype=torch.uint8, pin_memory=True).copy_(inp)
                s["out"] = torch.empty(inp.numel(), dtype=torch.uint8, pin_memory=True)
        return s
    if kind == "solve":
        ctx.gauge_upload(U, 18, P.F64)
        ctx.gauge_upload(U, case["links"], PREC[case["inner"]])
        if case["residual"] == "df64":
            ctx.gauge_upload(U, 18, P.DF64)
        s["b"] = _pack(ctx, _source(case, seed), "f64", case["nrhs"])
        s["x"] = torch.empty_like(s["b"])
        return s
    if kind == "load":
        n = case["nrhs"]
        s.update(U=U, phi=torch.view_as_real(_gauss(dims, n, _rng(seed, 1))), field=ctx.empty_full(P.F64, n))
        s["back"] = torch.empty_like(s["phi"])
        s["probe"] = _pack(ctx, _gauss(dims, 1, _rng(seed, 2)), case["prec"], 1)
        s["out"] = ctx.empty_half(PREC[case["prec"]])
        return s
    ctx.gauge_upload(U, 18, P.F64)
    s["bs"] = [_pack(ctx, _gauss(dims, 1, _rng(seed, 1 + k)), "f64", 1) for k in range(case["sources"])]
    s["xs"] = [torch.empty_like(b) for b in s["bs"]]
    return s


# ---------------------------------------------------------------- one pass


def _values(buf, prec):
    """The numbers of one packed half field."""
    if prec == "f64":
        return buf.view(torch.float64)
    if prec == "f32":
        return buf.view(torch.float32)
    sites = buf.numel() // 52
    return dict(halves=buf[: 48 * sites].view(torch.float16), norms=buf[48 * sites:].view(torch.float32))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        plq.cg_solve_batched(s["ctxs"], s["xs"], s["bs"], s["kappas"], inner_prec=PREC[case["inner"]])
        return [x.view(torch.float64) for x in s["xs"]]
    ctx = s["ctx"]
    if kind == "schur":
        ctx.schur_apply(s["out"], s["inp"], s["tmp"], 0.12, PREC[case["prec"]], dagger=case["dagger"])
        return _values(s["out"], case["prec"])
    if kind == "wilson":
        if case["mu"]:
            ctx.twisted_apply(s["out"], s["inp"], 0.12, case["mu"], PREC[case["prec"]])
        else:
            ctx.wilson_apply(s["out"], s["inp"], 0.12, PREC[case["prec"]])
        return _values(s["out"], case["prec"])
    if kind == "hop" and case["prec"] == "df64":
        # both parities, read back in double precision
        (ie, io), (oe, oo) = ctx.halves(s["inp"], P.DF64), ctx.halves(s["out"], P.DF64)
        ctx.hopping_eo(0, oe, io, P.DF64)
        ctx.hopping_eo(1, oo, ie, P.DF64)
        return ctx.unpack_spinor(s["values"], s["out"], P.DF64)
    if kind == "hop":
        ctx.hopping_eo(case["parity"], s["out"], s["inp"], PREC[case["prec"]], case["nrhs"])
        return _values(s["out"], case["prec"])
    if kind == "hop_host":
        ctx.hopping_eo_host(case["parity"], s["out"], s["inp"], PREC[case["prec"]], case["nrhs"])
        return _values(s["out"], case["prec"])
    if kind == "solve":
        kw = dict(inner_prec=PREC[case["inner"]], residual_prec=PREC[case["residual"]])
        if case["nrhs"] > 1:
            f = ctx.cg_solve_multi if case["method"] == "cg" else ctx.bicgstab_solve_multi
            f(s["x"], s["b"], case["kappa"], case["nrhs"], **kw)
        else:
            f = ctx.cg_solve if case["method"] == "cg" else ctx.bicgstab_solve
            f(s["x"], s["b"], case["kappa"], mu=case["mu"], **kw)
        return s["x"].view(torch.float64)
    if kind == "load":
        prec, n = PREC[case["prec"]], case["nrhs"]
        ctx.gauge_upload(s["U"], case["links"], prec)
        ctx.pack_spinor(s["field"], s["phi"], P.F64, n)
        ctx.unpack_spinor(s["back"], s["field"], P.F64, n)
        ctx.hopping_eo(0, s["out"], ctx.halves(s["probe"], prec)[1], prec)
        return dict(field=s["field"].view(torch.float64), back=s["back"], hop=_values(s["out"], case["prec"]))
    eig = plq.EigCG(ctx, case["nev"], case["m"], case["nev"] * case["sources"])
    for x, b in zip(s["xs"], s["bs"]):
        eig.solve(x, b, case["kappa"], tol=1e-11)
    eig.close()
    return [x.view(torch.float64) for x in s["xs"]]


# ---------------------------------------------------------------- the work of one pass


def _hop_work(V, prec, links, n):
    """Half-lattice application: input, output and the 8 links that touch each site once; 1320 flops a site."""
    Vh = V // 2
    return Vh * (2 * n * SITE_BYTES[prec] + 8 * links * REAL_BYTES[prec]), 1320.0 * Vh * n


def _solve_work(V, inner, links, n, method, iters):
    """`iters` iterations of the inner solver: its applications, and its vectors read and written once each."""
    b, f = _hop_work(V, inner, links, n)
    vec = (V // 2) * n * SITE_BYTES[inner]
    hops, moves = 4, 8  # CG on the normal equations and BiCGstab: two applications of two halves each
    if method == "bicgstab":
        moves = 12
    return iters * (hops * b + moves * vec), iters * (hops * f + (V // 2) * n * 24 * moves)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        per = [_solve_work(math.prod(d), case["inner"], case["links"], 1, "cg", 45) for d, _, _ in _batch_systems(case, 0)]
        return dict(bytes=sum(p[0] for p in per), flops=sum(p[1] for p in per))
    V = case["T"] * case["Lx"] * case["Ly"] * case["Lz"]
    if kind in ("hop", "hop_host"):
        b, f = _hop_work(V, case["prec"], case["links"], case["nrhs"])
        if case["prec"] == "df64":
            b, f = 2 * b + V * 2 * 192, 2 * f
        return dict(bytes=b, flops=f)
    if kind in ("schur", "wilson"):
        b, f = _hop_work(V, case["prec"], case["links"], 1)
        return dict(bytes=2 * b + (1 if kind == "schur" else 2) * (V // 2) * SITE_BYTES[case["prec"]], flops=2 * f)
    if kind == "solve":
        b, f = _solve_work(V, case["inner"], case["links"], case["nrhs"], case["method"],
                           50 if case["method"] == "cg" else 20)
        return dict(bytes=b, flops=f)
    if kind == "load":
        b, f = _hop_work(V, case["prec"], case["links"], 1)
        return dict(bytes=b + V * (576 + 4 * case["links"] * REAL_BYTES[case["prec"]] + case["nrhs"] * 4 * 192), flops=f)
    b, f = _solve_work(V, "f64", 18, 1, "cg", 60 * case["sources"])
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------- the same in 64 bits, in plain torch

# gamma_mu = [[0, A], [A^dagger, 0]]: (A v)_s = coef[s] v[perm[s]], for A and for A^dagger; the axis of mu in
# (n, T, Lz, Ly, Lx, 4, 3)
_GAMMA = [
    ((0, 1), (-1, -1), (-1, -1), 1),
    ((1, 0), (-1j, -1j), (1j, 1j), 4),
    ((1, 0), (-1, 1), (1, -1), 3),
    ((0, 1), (-1j, 1j), (1j, -1j), 2),
]


def _times(perm, coef, v):
    return torch.stack([coef[0] * v[..., perm[0], :], coef[1] * v[..., perm[1], :]], dim=-2)


def _shift(v, axis, by):
    """The field at x + by * mu (by = 1 or -1), antiperiodic in time."""
    w = torch.roll(v, -by, axis)
    if axis == 1:
        w[:, -1 if by > 0 else 0] *= -1
    return w


def _hop(U, phi):
    """Eq. (1) on (n, T, Lz, Ly, Lx, 4, 3)."""
    out = torch.zeros_like(phi)
    for mu, (perm, a, adag, axis) in enumerate(_GAMMA):
        u = U[..., mu, :, :]
        for by in (1, -1):
            if by > 0:  # U(x) (1 - gamma) phi(x + mu)
                p = _shift(phi, axis, 1)
                h = p[..., :2, :] - _times(perm, a, p[..., 2:, :])
                w = sum(u[..., None, :, b] * h[..., b, None] for b in range(3))
            else:  # U(x - mu)^dagger (1 + gamma) phi(x - mu)
                h = phi[..., :2, :] + _times(perm, a, phi[..., 2:, :])
                w = sum(u[..., None, b, :].conj() * h[..., b, None] for b in range(3))
                w = _shift(w, axis, -1)
            out[..., :2, :] += w
            out[..., 2:, :] -= by * _times(perm, adag, w)
    return out


def _wilson(U, phi, kappa, mu=0.0):
    out = phi - kappa * _hop(U, phi)
    if mu:
        out[..., :2, :] += 2j * kappa * mu * phi[..., :2, :]
        out[..., 2:, :] -= 2j * kappa * mu * phi[..., 2:, :]
    return out


def _dot(a, b):
    return (a.conj() * b).flatten(1).sum(1).view(-1, *([1] * (a.dim() - 1)))


def _solved(U, b, kappa, mu=0.0):
    """M x = b by BiCGstab, restarted from the residual until that is 1e-13 of b, each right-hand side for itself."""
    x = torch.zeros_like(b)
    nb = _dot(b, b).real.sqrt()
    for _ in range(8):
        r = b - _wilson(U, x, kappa, mu)
        n0 = _dot(r, r).real.sqrt()
        if bool((n0 <= 1e-13 * nb).all()):
            break
        # a random shadow residual: for a point source <r, r'> of the first step would vanish
        rhat = torch.randn(r.shape, dtype=r.dtype, device="cuda", generator=_rng(0, 63))
        p, d = r.clone(), torch.zeros_like(r)
        rho = _dot(rhat, r)
        for _ in range(300):
            v = _wilson(U, p, kappa, mu)
            alpha = rho / _dot(rhat, v)
            s = r - alpha * v
            t = _wilson(U, s, kappa, mu)
            omega = _dot(t, s) / _dot(t, t).real
            d += alpha * p + omega * s
            r = s - omega * t
            if bool((_dot(r, r).real.sqrt() <= 1e-7 * n0).all()):
                break
            new = _dot(rhat, r)
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
        x += d
    return x


def _half(psi, dims, parity):
    """The sites of one parity in checkerboard order: (Vh, n, 12) complex."""
    T, Lx, Ly, Lz = dims
    n = psi.shape[0]
    t, z, y = (torch.arange(k, device="cuda") for k in (T, Lz, Ly))
    odd = ((parity + t[:, None, None] + z[None, :, None] + y) % 2).bool()[None, :, :, :, None, None]
    v = psi.reshape(n, T, Lz, Ly, Lx // 2, 2, 12)
    return torch.where(odd, v[..., 1, :], v[..., 0, :]).reshape(n, -1, 12).transpose(0, 1)


def _laid_out(v, prec):
    """(Vh, n, 12) complex as the packed half field of `prec` holds it."""
    r = torch.view_as_real(v.contiguous())
    Vh, n = v.shape[:2]
    if prec == "f64":
        return r.permute(2, 0, 1, 3).contiguous()
    if prec == "f32":
        return r.reshape(Vh, n, 6, 4).permute(2, 0, 1, 3).contiguous()
    m = r.abs().amax(dim=(2, 3))
    q = r / m[..., None, None]
    return dict(halves=q.reshape(Vh, n, 3, 8).permute(2, 0, 1, 3).contiguous(), norms=m)


def _full64(psi, dims):
    return torch.cat([_laid_out(_half(psi, dims, p), "f64").reshape(-1) for p in (0, 1)])


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        got = []
        for k, (dims, kappa, eps) in enumerate(_batch_systems(case, seed)):
            g = _rng(seed, 2 + k)
            U = _links(dims, eps, g)
            got.append(_full64(_solved(U, _gauss(dims, 1, g), kappa), dims))
        return got
    dims = _dims(case)
    U = _links(dims, case.get("eps", 0.3), _rng(seed, 0))
    if kind in ("hop", "hop_host"):
        prec, n = case["prec"], case["nrhs"]
        phi = _gauss(dims, n, _rng(seed, 1))
        if prec == "df64":
            return _hop(U, phi)
        half = torch.empty((math.prod(dims) // 2, n, 12), dtype=torch.complex128, device="cuda")
        for r in range(n):
            half[:, r : r + 1] = _half(_hop(U, phi[r : r + 1]), dims, case["parity"])
        return _laid_out(half, prec)
    if kind == "schur":
        phi = _gauss(dims, 1, _rng(seed, 1))
        g5 = torch.tensor([1.0, 1, -1, -1], dtype=torch.float64, device="cuda")[:, None]
        parity = (sum(torch.arange(k, device="cuda").view([-1 if a == i else 1 for a in range(4)])
                      for i, k in enumerate(phi.shape[1:5])) % 2)[None, ..., None, None]
        e = torch.where(parity == 0, phi, torch.zeros_like(phi))
        v = g5 * e if case["dagger"] else e
        w = v - 0.12**2 * _hop(U, _hop(U, v))
        return _laid_out(_half(g5 * w if case["dagger"] else w, dims, 0), case["prec"])
    if kind == "wilson":
        psi = _wilson(U, _gauss(dims, 1, _rng(seed, 1)), 0.12, case["mu"])
        return torch.cat([_laid_out(_half(psi, dims, p), case["prec"]).reshape(-1) for p in (0, 1)])
    if kind == "solve":
        x = _solved(U, _source(case, seed), case["kappa"], case["mu"])
        return torch.cat([_laid_out(_half(x, dims, p), "f64").reshape(-1) for p in (0, 1)])
    if kind == "load":
        phi = _gauss(dims, case["nrhs"], _rng(seed, 1))
        field = torch.cat([_laid_out(_half(phi, dims, p), "f64").reshape(-1) for p in (0, 1)])
        hop = _hop(U, _gauss(dims, 1, _rng(seed, 2)))
        return dict(field=field, back=phi, hop=_laid_out(_half(hop, dims, 0), case["prec"]))
    return [_full64(_solved(U, _gauss(dims, 1, _rng(seed, 1 + k)), case["kappa"]), dims) for k in range(case["sources"])]
