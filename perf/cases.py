"""Timed workloads of the library, each through its public entry points.

A case is a dict with a "kind":

* ``apply``    gdr_op_apply on a Wilson operator: the matvec a program calls for its own Krylov
               steps (complex64, gauge links in complex64 or bf16) and for true residuals (FP64);
* ``csr``      gdr_op_apply on a ragged batch of convection-diffusion matrices (one: a single matrix);
* ``cycle``    gdr_arnoldi_cycle: one Arnoldi cycle, from one vector or continued from a kept pair;
* ``reduced``  gdr_dense_gmres_sh: the small multi-shift solve at the end of a cycle;
* ``dot``, ``resid``  gdr_basis_dot, gdr_basis_residual_update: the projection of many residuals over
               one kept basis;
* ``restart``  gdr_basis_update: a cycle's basis rotated onto the kept vectors (with the solution
               update in FP64);
* ``solve``    gdr_solve_multishift: a whole solve, to eleven digits, so that the solution itself is
               good to the digits an FP64 result is compared at.

Wilson lattices run from 4^4 to 24^3x32, the basis from 20 to 81 vectors, batches from one column to
ten shifts times twelve right-hand sides.  Everything is called as the defaults give it: no launch
shape is tuned first.

Results that the complex64 path leaves in an FP64 buffer (Hbar of a complex64 cycle, the projection's
dots) carry the accuracy of the complex64 vectors that they come from; the program that goes on with
them in that precision takes them as complex64, and so does ``run``.
"""
import math
import weakref

import numpy as np
import torch

import paper_0707_0502_gb300 as g

#: critical kappa of the synthetic links by their spread eps (workloads/kappa_c.json)
KAPPA_C = {0.3: 0.13254, 0.4: 0.13885, 0.5: 0.14769}
C64, C128 = torch.complex64, torch.complex128


def listed():
    return [
        # one Krylov step of a program's own solver on a medium lattice: launches and latency count
        dict(name="apply_c64_16^4_x1", kind="apply", L="16x16x16x16", prec="c64", links="c64", ncol=1),
        # the batched matvec of twelve right-hand sides on the largest lattice, links in bf16
        dict(name="apply_bf16_24^3x32_x12", kind="apply", L="24x24x24x32", prec="c64", links="bf16", ncol=12),
        # FP64 true residuals of the eight shifts of one right-hand side
        dict(name="apply_fp64_16^4_x8", kind="apply", L="16x16x16x16", prec="fp64", links="c64", ncol=8),
        # the operator of the batch of 64 independent problems of uneven size (sides 32 to 256)
        dict(name="csr_batch64_c64", kind="csr", nprob=64, side_lo=32, side_hi=256, prec="c64"),
        # the first cycle of GMRES-DR(80, .) on the largest lattice: Gram-Schmidt against HBM
        dict(name="cycle_c64_24^3x32_m80", kind="cycle", L="24x24x24x32", prec="c64", links="bf16", j0=0, m=80),
        # an FP64 cycle of GMRES-DR(60,30) after a restart: the plain FP64 solve and the clean-up stage
        dict(name="cycle_fp64_16^4_30_60", kind="cycle", L="16x16x16x16", prec="fp64", links="c64", j0=30, m=60),
        # the reduced multi-shift solve of GMRES-DR(40,20), the smallest call: latency alone
        dict(name="reduced_m40_x6", kind="reduced", m=40, k=20, ns=6),
        # the projection of 8 shifts x 8 right-hand sides over a kept basis of 31 vectors
        dict(name="dot_16^4_31x64", kind="dot", L="16x16x16x16", prec="c64", nv=31, ncol=64),
        # its residual update at 10 shifts x 12 right-hand sides on the largest lattice
        dict(name="resid_24^3x32_41x120", kind="resid", L="24x24x24x32", prec="c64", nv=41, ncol=120),
        # the restart of GMRES-DR(80,40) on the largest lattice
        dict(name="restart_c64_24^3x32_81_41", kind="restart", L="24x24x24x32", prec="c64", nv=81, nout=41, nx=0),
        # a whole mixed solve of one right-hand side on the small lattice: a chain of short launches
        dict(name="solve_8^4_6x1", kind="solve", L="8x8x8x8", eps=0.3, prec="c64", links="c64", ns=6, nrhs=1,
             m=40, k=20, m_proj=20),
        # a whole mixed solve, 8 shifts x 8 right-hand sides on the medium lattice
        dict(name="solve_16^4_8x8", kind="solve", L="16x16x16x16", eps=0.4, prec="c64", links="c64", ns=8, nrhs=8,
             m=60, k=30, m_proj=30),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_lattice(rng, lo, hi, most):
    """Extents lo to hi, the time extent up to twice the others', at most `most` sites."""
    while True:
        s = _log_int(rng, lo, hi)
        d = [max(2, s + rng.choice((0, 0, 0, -1, 1))) for _ in range(3)] + [_log_int(rng, max(2, s // 2), 2 * s)]
        if math.prod(d) <= most:
            return "x".join(map(str, d))


def draw(rng):
    kind = rng.choice(("apply", "apply", "apply", "csr", "cycle", "cycle", "reduced", "dot", "resid", "restart",
                       "solve", "solve"))
    if kind == "apply":
        prec = rng.choice(("c64", "c64", "fp64"))
        return dict(kind=kind, L=_draw_lattice(rng, 4, 24, 442368), prec=prec, links=rng.choice(("c64", "bf16")),
                    ncol=_log_int(rng, 1, 12))
    if kind == "csr":
        lo = _log_int(rng, 32, 128)
        return dict(kind=kind, nprob=_log_int(rng, 1, 64), side_lo=lo, side_hi=_log_int(rng, lo, 256),
                    prec=rng.choice(("c64", "fp64")))
    if kind == "cycle":
        prec = rng.choice(("c64", "c64", "fp64"))
        m = rng.randint(20, 80)
        return dict(kind=kind, L=_draw_lattice(rng, 4, 16, 65536), prec=prec, links=rng.choice(("c64", "bf16")),
                    j0=rng.choice((0, m // 2)), m=m)
    if kind == "reduced":
        m = rng.randint(20, 80)
        return dict(kind=kind, m=m, k=m // 2, ns=rng.randint(1, 12))
    if kind in ("dot", "resid"):
        prec = rng.choice(("c64", "c64", "c64", "fp64"))
        most = 442368 if prec == "c64" else 65536
        return dict(kind=kind, L=_draw_lattice(rng, 6, 24, most), prec=prec, nv=rng.randint(11, 48),
                    ncol=_log_int(rng, 2, 120 if prec == "c64" else 16))
    if kind == "restart":
        prec = rng.choice(("c64", "c64", "fp64"))
        nv = rng.randint(21, 81)
        return dict(kind=kind, L=_draw_lattice(rng, 4, 24, 442368 if prec == "c64" else 65536), prec=prec, nv=nv,
                    nout=nv // 2, nx=0 if prec == "c64" else rng.randint(1, 8))
    prec = rng.choice(("c64", "c64", "c64", "fp64"))
    m = rng.randint(25, 60)
    return dict(kind=kind, L=_draw_lattice(rng, 4, 12 if prec == "c64" else 6, 20736 if prec == "c64" else 1500),
                eps=rng.choice((0.3, 0.4)), prec=prec, links="c64", ns=rng.randint(1, 8),
                nrhs=_log_int(rng, 1, 8 if prec == "c64" else 2), m=m, k=m // 2, m_proj=m - m // 2)


# ------------------------------------------------------------------ inputs

_CTX = []


def _ctx():
    """The program's one library context."""
    if not _CTX:
        _CTX.append(g.gdr_create(0))
    return _CTX[0]


class _State(dict):
    """A case's inputs and handles; the operator goes with it."""

    def own(self, op):
        self["op"] = op
        weakref.finalize(self, g.gdr_op_destroy, op)


def _dims(case):
    return tuple(int(x) for x in case["L"].split("x"))


def _sites(case):
    return math.prod(_dims(case))


def _prec(case):
    return g.GDR_PREC_FP64 if case["prec"] == "fp64" else g.GDR_PREC_MIXED


def _dtype(case):
    return C128 if case["prec"] == "fp64" else C64


def _gen(seed):
    return torch.Generator("cuda").manual_seed(int(seed))


def _randn(gen, *shape, dtype=C128):
    return torch.randn(*shape, dtype=dtype, device="cuda", generator=gen)


def _links(case, gen):
    """SU(3) links exp(i eps X), X = sum_a omega_a lambda_a / 2 with omega_a ~ N(0,1), [4, V, 3, 3]."""
    lam = np.zeros((8, 3, 3), dtype=np.complex128)
    for a, (p, q) in enumerate(((0, 1), (0, 2), (1, 2))):
        lam[2 * a, p, q] = lam[2 * a, q, p] = 1
        lam[2 * a + 1, p, q], lam[2 * a + 1, q, p] = -1j, 1j
    lam[6] = np.diag([1, -1, 0])
    lam[7] = np.diag([1, 1, -2]) / math.sqrt(3)
    eps = case.get("eps", 0.5 if case.get("links") == "bf16" else 0.4)
    omega = torch.randn(4 * _sites(case), 8, dtype=torch.float64, device="cuda", generator=gen)
    X = (omega.to(C128) @ torch.as_tensor(lam.reshape(8, 9), device="cuda")).reshape(-1, 3, 3)
    M = (0.5j * eps / 8) * X
    U = torch.eye(3, dtype=C128, device="cuda") + M / 14
    for i in range(13, 0, -1):  # Taylor series of exp(M) by Horner, M scaled by 1/8
        U = torch.eye(3, dtype=C128, device="cuda") + (M @ U) / i
    for _ in range(3):
        U = U @ U
    return U.reshape(4, -1, 3, 3).contiguous()


def _wilson_op(case, U):
    return g.gdr_op_wilson(_ctx(), _dims(case), U, 0.0, g.GDR_LINK_BF16 if case["links"] == "bf16" else g.GDR_LINK_C64)


def _shifts(eps, count):
    """-1 / kappa for kappa from 0.97 kappa_c (the base system) down to 0.115."""
    return -1.0 / np.linspace(0.97 * KAPPA_C[eps], 0.115, count) + 0j


def _z2(gen, *shape):
    re = torch.randint(0, 2, shape, device="cuda", generator=gen, dtype=torch.int8)
    im = torch.randint(0, 2, shape, device="cuda", generator=gen, dtype=torch.int8)
    return torch.complex(re.double() * 2 - 1, im.double() * 2 - 1) / math.sqrt(2)


def _convdiff(side, cx, cy, delta):
    """Five-point convection-diffusion on the unit square, CSR, rows in lexicographic order."""
    h = 1.0 / (side + 1)
    iy, ix = np.divmod(np.arange(side * side), side)
    nb = [(0, -1, -1 / h**2 - cy / (2 * h)), (-1, 0, -1 / h**2 - cx / (2 * h)), (0, 0, 4 / h**2 + 1j * delta),
          (1, 0, -1 / h**2 + cx / (2 * h)), (0, 1, -1 / h**2 + cy / (2 * h))]
    ok = np.stack([(ix + a >= 0) & (ix + a < side) & (iy + b >= 0) & (iy + b < side) for a, b, _ in nb], 1)
    col = np.stack([(iy + b) * side + ix + a for a, b, _ in nb], 1)
    val = np.broadcast_to(np.array([v for _, _, v in nb]), ok.shape)
    rowptr = np.concatenate([[0], np.cumsum(ok.sum(1))])
    return rowptr.astype(np.int32), col[ok].astype(np.int32), val[ok].astype(np.complex128)


def _csr_inputs(case, seed):
    r = np.random.default_rng([int(seed), 5])
    sides = np.linspace(case["side_hi"], case["side_lo"], case["nprob"]).round().astype(int)
    sides = np.concatenate([sides[::2], sides[1::2]])  # uneven neighbours
    mats = [_convdiff(int(s), r.uniform(-20, 20), r.uniform(-20, 20), r.uniform(0, 0.5)) for s in sides]
    n = int(max(sides)) ** 2
    X = _randn(_gen(seed), case["nprob"], n, dtype=_dtype(case))
    for p, s in enumerate(sides):  # a problem's column is zero behind its own rows
        X[p, int(s) ** 2:] = 0
    sigma = np.resize(np.array([1.0, 0.0, 0.1, 0.5]), case["nprob"]) + 0j
    return mats, X, sigma


def _reduced_inputs(case, seed):
    """Hbar as after a restart (a full leading block, Hessenberg behind it), c = ||r|| e_1 rotated, shifts, beta."""
    m, k, ns = case["m"], case["k"], case["ns"]
    r = np.random.default_rng([int(seed), 6])
    H = np.triu(r.standard_normal((m + 1, m)) + 1j * r.standard_normal((m + 1, m)), -1)
    H[: k + 1, :k] = r.standard_normal((k + 1, k)) + 1j * r.standard_normal((k + 1, k))
    H *= 8.0 / math.sqrt(m)  # the hopping term's range: a cycle reduces the residual by a few digits
    H[np.arange(1, m + 1), np.arange(m)] += 6.0
    c = np.zeros(m + 1, dtype=complex)
    c[: k + 1] = r.standard_normal(k + 1) + 1j * r.standard_normal(k + 1)
    beta = r.standard_normal(ns) + 1j * r.standard_normal(ns)
    beta[0] = 1.0
    return H, c, _shifts(0.3, ns), beta


def _small(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _hop_tables(case, U):
    """The links as the entry point holds them, in 64 bits, forward and backward, with each direction's axis."""
    Lx, Ly, Lz, Lt = _dims(case)
    if case["prec"] != "fp64":
        u = torch.view_as_real(U).float()
        u = u.bfloat16().double() if case["links"] == "bf16" else u.double()
        U = torch.view_as_complex(u.contiguous())
    f = U.reshape(4, Lt, Lz, Ly, Lx, 3, 3)
    return [(f[mu], torch.roll(f[mu], 1, 3 - mu).conj().transpose(-1, -2).contiguous(), 3 - mu) for mu in range(4)]


#: gamma_x, y, z, t in the chiral basis: (gamma psi)_s = phase_s psi_perm(s)
_GAMMA = (((3, 2, 1, 0), (-1j, -1j, 1j, 1j)), ((3, 2, 1, 0), (-1, 1, 1, -1)), ((2, 3, 0, 1), (-1j, 1j, 1j, -1j)),
          ((2, 3, 0, 1), (1, 1, 1, 1)))


def _wilson_matvec(case, tables, x, sigma):
    """-(H + sigma) x in 64 bits, by rolled fields."""
    Lx, Ly, Lz, Lt = _dims(case)
    psi = x.reshape(Lt, Lz, Ly, Lx, 4, 3)
    out = torch.zeros_like(psi)
    for (fwd, bwd, ax), (perm, phase) in zip(tables, _GAMMA):
        ph = torch.tensor(phase, dtype=C128, device=x.device)[:, None]
        for step, u, sign in ((-1, fwd, -1), (1, bwd, 1)):
            h = torch.roll(psi, step, ax)
            h = sum(h[..., :, b, None] * u[..., None, :, b] for b in range(3))
            out += h + sign * ph * h[..., list(perm), :]
    return -out.reshape(-1) - sigma * x


def _arnoldi(case, U, V, H, j0, m):
    """Arnoldi steps j0..m-1 in 64 bits, Gram-Schmidt twice, rows of V the vectors."""
    t = _hop_tables(case, U)
    for j in range(j0, m):
        w = _wilson_matvec(case, t, V[j], 0)
        for _ in range(2):
            h = V[: j + 1].conj() @ w
            w = w - h @ V[: j + 1]
            H[j, : j + 1] += h
        H[j, j + 1] = torch.linalg.vector_norm(w)
        V[j + 1] = w / H[j, j + 1]


def _cycle_inputs(case, seed):
    """The links and V, Hbar with their given columns in 64 bits: a Z2 start vector, or j0 steps from it."""
    gen = _gen(seed)
    n = 12 * _sites(case)
    U = _links(case, gen)
    v = _z2(gen, n)
    V = torch.zeros(case["j0"] + 1, n, dtype=C128, device="cuda")
    V[0] = v / torch.linalg.vector_norm(v)
    H = torch.zeros(case["m"], case["m"] + 1, dtype=C128, device="cuda")
    _arnoldi(case, U, V, H, 0, case["j0"])
    return U, V.to(_dtype(case)), H


def _orthonormal(gen, nv, n, dtype):
    V = _randn(gen, nv, n, dtype=dtype)
    return V / torch.linalg.vector_norm(V, dim=1, keepdim=True)


def _basis_inputs(case, seed):
    gen = _gen(seed)
    n, nv = 12 * _sites(case), case["nv"]
    V = _orthonormal(gen, nv, n, _dtype(case))
    if case["kind"] == "restart":
        C = torch.linalg.qr(_randn(gen, nv, case["nout"]))[0]
        D = _randn(gen, nv, case["nx"]) / math.sqrt(nv)
        X = _randn(gen, case["nx"], n) if case["nx"] else None
        return V, torch.cat([C, D], 1).T.contiguous(), X
    return V, _randn(gen, case["ncol"], n, dtype=_dtype(case)), _randn(gen, case["ncol"], nv)


def prepare(case, seed):
    s, kind = _State(case=case), case["kind"]
    ctx = _ctx()
    if kind == "apply":
        gen, n = _gen(seed), 12 * _sites(case)
        s.own(_wilson_op(case, _links(case, gen)))
        s["X"] = _randn(gen, case["ncol"], n, dtype=_dtype(case))
        s["Y"] = torch.empty_like(s["X"])
        s["sigma"] = _shifts(0.4, case["ncol"])
    elif kind == "csr":
        mats, s["X"], s["sigma"] = _csr_inputs(case, seed)
        s["Y"] = torch.zeros_like(s["X"])
        s.own(g.gdr_op_csr_batch(ctx, [len(a[0]) - 1 for a in mats], [len(a[1]) for a in mats],
                                 *(_small(np.concatenate([a[i] for a in mats])) for i in range(3))))
    elif kind == "cycle":
        U, V, s["H"] = _cycle_inputs(case, seed)
        s.own(_wilson_op(case, U))
        s["V"] = torch.zeros(case["m"] + 1, V.shape[1], dtype=V.dtype, device="cuda")
        s["V"][: case["j0"] + 1] = V
    elif kind == "reduced":
        H, c, s["sigma"], beta = _reduced_inputs(case, seed)
        m, ns = case["m"], case["ns"]
        s["H"], s["c"], s["beta"] = _small(H.T), _small(c), _small(beta)
        s["out"] = [torch.empty(ns, m, dtype=C128, device="cuda"), torch.empty(m + 1, dtype=C128, device="cuda"),
                    torch.empty(ns, dtype=C128, device="cuda"), torch.empty(ns, dtype=torch.float64, device="cuda")]
    elif kind in ("dot", "resid"):
        s["V"], s["R"], s["T"] = _basis_inputs(case, seed)
        s["C"] = torch.empty(case["ncol"], case["nv"], dtype=C128, device="cuda")
    elif kind == "restart":
        s["V"], s["C"], s["X"] = _basis_inputs(case, seed)
    else:
        gen, n = _gen(seed), 12 * _sites(case)
        s.own(_wilson_op(case, _links(case, gen)))
        s["B"] = _z2(gen, case["nrhs"], n)
        s["X"] = torch.empty(case["nrhs"], case["ns"], n, dtype=C128, device="cuda")
        s["sigma"] = _shifts(case["eps"], case["ns"])
        s["params"] = g.gdr_params_default(m=case["m"], k=case["k"], m_proj=case["m_proj"], tol=1e-11, prec=_prec(case),
                                           refine_max=6)
    return s


def run(s):
    case, ctx = s["case"], _ctx()
    kind = case["kind"]
    if kind in ("apply", "csr"):
        g.gdr_op_apply(ctx, s["op"], _prec(case), s["sigma"], s["X"], s["Y"])
        return s["Y"]
    if kind == "cycle":
        g.gdr_arnoldi_cycle(ctx, s["op"], _prec(case), s["V"], case["j0"], case["m"], s["H"])
        return {"V": s["V"], "H": s["H"] if case["prec"] == "fp64" else s["H"].to(C64)}
    if kind == "reduced":
        g.gdr_dense_gmres_sh(ctx, case["m"], s["sigma"], s["H"], s["c"], s["beta"], *s["out"])
        return s["out"]
    if kind == "dot":
        g.gdr_basis_dot(ctx, _prec(case), s["V"].shape[1], case["nv"], s["V"], case["ncol"], s["R"], s["R"].shape[1],
                        s["C"])
        return s["C"] if case["prec"] == "fp64" else s["C"].to(C64)
    if kind == "resid":
        g.gdr_basis_residual_update(ctx, _prec(case), s["V"].shape[1], case["nv"], s["V"], case["ncol"], s["T"], s["R"],
                                    s["R"].shape[1])
        return s["R"]
    if kind == "restart":
        g.gdr_basis_update(ctx, _prec(case), s["V"].shape[1], case["nv"], s["V"], s["C"], case["nout"], case["nx"],
                           s["X"])
        return [s["V"], s["X"]]
    status, _, _ = g.gdr_solve_multishift(ctx, s["op"], s["sigma"], s["B"], s["X"], s["params"])
    if status != g.GDR_OK:
        raise RuntimeError("not converged")
    return s["X"]


# ------------------------------------------------------------------ what a pass needs at least

def work(case):
    kind = case["kind"]
    if kind == "csr":
        r = (case["side_lo"] + case["side_hi"]) / 2
        rows, sv = case["nprob"] * r * r, 16 if case["prec"] == "fp64" else 8
        return {"bytes": rows * (5 * (sv + 4) + 4 + 2 * sv), "flops": rows * 5 * 8}
    if kind == "reduced":
        m, ns = case["m"], case["ns"]
        return {"bytes": 16.0 * ((m + 1) * m + ns * m + 2 * (m + 1) + 3 * ns), "flops": ns * 8 * 2 / 3 * m**3}
    n = 12 * _sites(case)
    sv = 16 if case["prec"] == "fp64" else 8
    sl = 16 if case["prec"] == "fp64" else 4 if case.get("links") == "bf16" else 8
    mat = lambda c: (36 * sl * n / 12 + 2 * c * n * sv, 1368 * c * n / 12)  # noqa: E731
    if kind == "apply":
        b, f = mat(case["ncol"])
        return {"bytes": b, "flops": f}
    if kind == "cycle":  # each step reads the basis for its projection and for its update
        j0, m = case["j0"], case["m"]
        vecs = sum(j + 1 for j in range(j0, m))
        b, f = mat(1)
        return {"bytes": (m - j0) * b + 2 * vecs * n * sv, "flops": (m - j0) * f + 4 * vecs * 8 * n}
    if kind == "dot":
        return {"bytes": (case["nv"] + case["ncol"]) * n * sv, "flops": 8 * case["nv"] * case["ncol"] * n}
    if kind == "resid":
        return {"bytes": (case["nv"] + 2 * case["ncol"]) * n * sv, "flops": 8 * case["nv"] * case["ncol"] * n}
    if kind == "restart":
        outs = case["nout"] + case["nx"]
        return {"bytes": (case["nv"] + case["nout"]) * n * sv + 2 * case["nx"] * n * 16,
                "flops": 8 * case["nv"] * outs * n}
    # a solve: one cycle for the first right-hand side and one projected cycle for each pair after it
    c = dict(case, kind="cycle", j0=0)
    first, pair = work(c), work(dict(c, m=case["m_proj"]))
    pairs = case["ns"] * case["nrhs"]
    return {q: first[q] + pairs * pair[q] for q in ("bytes", "flops")}


# ------------------------------------------------------------------ the same in 64 bits

def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        gen, n = _gen(seed), 12 * _sites(case)
        t = _hop_tables(case, _links(case, gen))
        X = _randn(gen, case["ncol"], n, dtype=_dtype(case)).to(C128)
        return torch.stack([_wilson_matvec(case, t, x, s) for x, s in zip(X, _shifts(0.4, case["ncol"]).tolist())])
    if kind == "csr":
        mats, X, sigma = _csr_inputs(case, seed)
        Y, X = np.zeros(tuple(X.shape), dtype=complex), X.to(C128).cpu().numpy()
        for p, (rowptr, col, val) in enumerate(mats):
            n = len(rowptr) - 1
            val = val if case["prec"] == "fp64" else val.astype(np.complex64).astype(complex)
            Y[p, :n] = np.add.reduceat(val * X[p, col], rowptr[:-1]) - sigma[p] * X[p, :n]
        return Y
    if kind == "cycle":
        U, V0, H = _cycle_inputs(case, seed)
        V = torch.zeros(case["m"] + 1, V0.shape[1], dtype=C128, device="cuda")
        V[: case["j0"] + 1] = V0.to(C128)
        _arnoldi(case, U, V, H, case["j0"], case["m"])
        return {"V": V, "H": H}
    if kind == "reduced":
        H, c, sigma, beta = _reduced_inputs(case, seed)
        I = np.eye(case["m"] + 1, case["m"])
        d = np.linalg.lstsq(H - sigma[0] * I, c, rcond=None)[0]
        s = c - (H - sigma[0] * I) @ d
        D, beta_new = [d], [1.0]
        for sg, b in zip(sigma[1:], beta[1:]):
            y = np.linalg.solve(np.concatenate([H - sg * I, s[:, None]], 1), b * c)
            D.append(y[:-1])
            beta_new.append(y[-1])
        rn = np.linalg.norm(s)
        return [np.stack(D), s, np.array(beta_new) + 0j, np.abs(beta_new) * rn]
    if kind == "dot":
        V, R, _ = _basis_inputs(case, seed)
        C = torch.zeros(case["ncol"], case["nv"], dtype=C128, device="cuda")
        for q in range(0, V.shape[1], 1 << 20):
            C += R[:, q:q + (1 << 20)].to(C128) @ V[:, q:q + (1 << 20)].to(C128).conj().T
        return C
    if kind == "resid":
        V, R, T = _basis_inputs(case, seed)
        return torch.stack([r.to(C128) + t @ V.to(C128) for r, t in zip(R, T)]) if R.shape[1] * case["ncol"] < 1 << 27 \
            else R.to(C128).addmm_(T, V.to(C128))
    if kind == "restart":
        V, C, X = _basis_inputs(case, seed)
        V = V.to(C128)
        out = C @ V
        V[: case["nout"]] = out[: case["nout"]]
        return [V, None if X is None else X + out[case["nout"]:]]
    return None
