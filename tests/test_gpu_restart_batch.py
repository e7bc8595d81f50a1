"""The tensor-core restart of a batch: bases of their own lengths (runs on a GB300; -m gpu).

GMRES-DR(60, 30) with four shifts rotates 61 vectors onto 31 and updates four solutions: 35
outputs, on the tensor cores, one batch column per problem.  Problem sizes: one to 31 row tiles
of 64 and 0 to 41 rows over, odd and even, the last tile a single row (961) or whole (1600);
the small problems end a cycle or more before the others and must be left alone.

A wrong row, column or neighbour shows in the residuals after the complex64 stage, which nothing
refines here: the recurrence stops a problem at 1e-7 and the true residuals are then held to
four times what the CUDA-core restart leaves (the same rounding, drawn again)."""
import numpy as np
import pytest

import workloads as W
from oracle import CSROperator, gmres_dr_sh

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_0707_0502_gb300 as g  # noqa: E402


def _problems():
    gen = np.random.default_rng([61, 3])
    out = []
    for s in (9, 45, 11, 31, 13, 40, 17, 22, 25):
        rowptr, col, vals = W.convdiff_csr(s, *gen.uniform(-20, 20, 2), gen.uniform(0, 0.5))
        out.append(W.Problem(name=f"cd{s}", op=("csr", rowptr, col, vals), n=s * s,
                             sigma=np.array([1.0, 0.0, 0.1, 0.5], complex), B=W.gaussian_complex(gen, s * s, 1), m=60,
                             k=30, m_proj=30))
    return out


def _solve(ctx, probs, flags):
    op = g.make_batch_operator(ctx, probs)
    B = torch.as_tensor(np.concatenate([p.B[:, 0] for p in probs])).cuda()
    X = torch.zeros(4 * len(B), dtype=torch.complex128, device="cuda")
    prm = g.gdr_params_default(m=60, k=30, m_proj=30, tol=1e-8, inner_tol=1e-7, prec=g.GDR_PREC_MIXED, flags=flags)
    st, rep, per = g.gdr_solve_batch(ctx, op, np.stack([p.sigma for p in probs]), B, X, prm)
    g.gdr_op_destroy(op)
    Xh, off, out = X.cpu().numpy(), 0, []
    for p in probs:
        out.append(Xh[4 * off: 4 * (off + p.n)].reshape(4, p.n))
        off += p.n
    return st, rep, per, out


def _residuals(probs, X):
    r = []
    for p, x in zip(probs, X):
        A = CSROperator(*p.op[1:])
        b = p.B[:, 0]
        r.append([np.linalg.norm(b - A.matvec(xi) + s * xi) / np.linalg.norm(b) for xi, s in zip(x, p.sigma)])
    return np.array(r)


def test_ragged_batch():
    import __graft_entry__
    __graft_entry__.build()
    ctx = g.gdr_create(0)
    probs = _problems()
    g.gdr_profile(ctx, True)
    st, rep, per, X = _solve(ctx, probs, 0)
    prof = g.gdr_profile_report(ctx)
    g.gdr_profile(ctx, False)
    assert st == g.GDR_OK and (per == 0).all(), (rep, per)
    assert prof["tc_restart_c64"]["launches"] >= 2 and "combine_restart_c64" not in prof
    assert rep["cycles_rhs1"] >= 2
    assert _residuals(probs, X).max() <= 1e-8
    for p, x in zip(probs, X):
        if p.n <= 300:
            ref = gmres_dr_sh(CSROperator(*p.op[1:]).matvec, p.B[:, 0], p.sigma, p.m, p.k, 1e-12)["x"]
            assert np.linalg.norm(x - ref.T) <= 1e-6 * np.linalg.norm(ref), p.name
    stage = g.GDR_FLAG_NO_REFINE
    tc = _residuals(probs, _solve(ctx, probs, stage)[3])
    plain = _residuals(probs, _solve(ctx, probs, stage | g.GDR_FLAG_NO_TENSOR_CORES)[3])
    assert (tc <= 4 * np.maximum(plain, plain.max(1, keepdims=True))).all(), (tc, plain)
    g.gdr_destroy(ctx)
