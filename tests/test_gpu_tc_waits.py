"""A tensor-core wait that gives up in a call that does not synchronise is reported by the next
one that does (runs on a GB300; -m gpu).

The self-test's kernel waits about a second for an arrival that never comes and leaves the mark
that gdr_basis_update would: every synchronising entry point returns GDR_ETIMEOUT once, with
its own results complete, and the one after it is clean."""
import numpy as np
import pytest

from tests.gpu_util import dev, small_wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_0707_0502_gb300 as g  # noqa: E402


def test_reported_by_the_next_synchronising_call():
    import __graft_entry__
    __graft_entry__.build()
    ctx = g.gdr_create(0)
    p, _ = small_wilson(dims=(2, 2, 2, 2), nshift=2, nrhs=2)
    op = g.make_operator(ctx, p)
    r = np.random.default_rng(0)
    n, m, k = p.n, 6, 2
    c128 = lambda *s: torch.zeros(s, dtype=torch.complex128, device="cuda")
    rnd = lambda *s: dev(r.standard_normal(s) + 1j * r.standard_normal(s))
    V, H = c128(m + 1, n), c128(m, m + 1)
    V[0] = rnd(n)
    V[0] /= torch.linalg.vector_norm(V[0])
    B, X = dev(p.B.T), c128(2, 2, n)
    prm = g.gdr_params_default(m=p.m, k=p.k, m_proj=p.m_proj, tol=1e-8, prec=g.GDR_PREC_MIXED)
    _, _, defl = g.gdr_solve_multishift(ctx, op, p.sigma, B, X, prm, want_defl=True)
    assert defl
    Hd, c, one, s, bn = rnd(m, m + 1), rnd(m + 1), dev(np.ones(2, complex)), c128(m + 1), c128(2)
    Hu = torch.tril(Hd, 1)  # row j is column j of a Hessenberg matrix
    D, nrm, f = c128(2, m), torch.zeros(2, dtype=torch.float64, device="cuda"), g.GDR_PREC_FP64
    C = c128(9, k)
    calls = {
        "cycle": lambda: g.gdr_arnoldi_cycle(ctx, op, f, V, 0, m, H),
        "step": lambda: g.gdr_arnoldi_step(ctx, op, f, V, 1, c128(3)),
        "gmres_sh": lambda: g.gdr_dense_gmres_sh(ctx, m, [0, 1], Hd, c, one, D, s, bn, nrm),
        "noalloc": lambda: g.gdr_dense_gmres_sh_noalloc(ctx, m, [0, 1], Hd, c, one, D, s, bn, nrm),
        "ls": lambda: g.gdr_dense_ls(ctx, f, m, 0, Hu, c, c128(m), s),
        "restart": lambda: g.gdr_dense_restart(ctx, f, m, k, 0, Hd, s, c128(m), c128(k + 1, m + 1), c128(k, k + 1),
                                               c128(k + 1)),
        "dot": lambda: g.gdr_basis_dot(ctx, f, n, k, V, 9, rnd(9, n), n, C),
        "resid": lambda: g.gdr_basis_residual_update(ctx, f, n, k, V, 9, rnd(9, k), rnd(9, n), n),
        "solve": lambda: g.gdr_solve_multishift(ctx, op, p.sigma, B, X, prm),
        "proj": lambda: g.gdr_solve_proj(ctx, op, defl, p.sigma, B, X, prm),
        "export": lambda: g.gdr_defl_export(ctx, defl),
        "autotune": lambda: g.gdr_autotune(ctx, op, f, 1),
        "profile": lambda: g.gdr_profile(ctx, False),
        "report": lambda: g.gdr_profile_report(ctx),
        "barrier": lambda: g._check(g.gdr_barrier_selftest(ctx, 1, 0), ctx),
    }
    for name, call in calls.items():
        call()
        want = D.clone(), s.clone(), V.clone(), C.clone()
        g.gdr_tc_wait_selftest(ctx)
        with pytest.raises(g.GdrError) as e:
            call()
        assert e.value.status == g.GDR_ETIMEOUT, name
        torch.cuda.synchronize()
        if name in ("cycle", "gmres_sh", "noalloc", "ls", "restart"):
            for a, b in zip((D, s, V), want):
                assert torch.equal(a, b), name
        call()
    g.gdr_defl_destroy(defl)
    g.gdr_op_destroy(op)
    g.gdr_destroy(ctx)
