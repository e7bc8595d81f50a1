"""The reduced multi-shift solve's QR at the edges of its column mapping (runs on a GB300; -m gpu).

A reflector gives each column 4, 8 or 16 lanes of a 128-thread block, as many as keep all
remaining columns in one pass, up to four passes of 32 columns.  m = 1 (one reflector), 6 / 7 /
8 and 14 / 15 / 16 columns (where the lane count changes with the last ones), 31 (one pass of
32), 32, 64 and 96 (two, three, four passes).  Against numpy's FP64 solve of the same systems,
relative to the norm of each result: 1e-13 times the condition number of the system (backward
error of Householder QR, a modest multiple of m 2^-53).  Two to eight shifts are one cluster
of as many CTAs, whose shifts apply the kept reflectors to the base solve's residual; one and
nine shifts take the two launches."""
import numpy as np
import pytest

from tests.gpu_util import dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_0707_0502_gb300 as g  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = g.gdr_create(0)
    yield c
    g.gdr_destroy(c)


@pytest.mark.parametrize("m,ns", [(m, 3) for m in (1, 2, 6, 7, 8, 14, 15, 16, 31, 32, 64, 96)] +
                         [(33, 1), (33, 2), (33, 8), (33, 9), (95, 8)])
def test_reduced_solve_sizes(ctx, m, ns):
    r = np.random.default_rng(m)
    H = (r.standard_normal((m + 1, m)) + 1j * r.standard_normal((m + 1, m))) / np.sqrt(m)
    c = r.standard_normal(m + 1) + 1j * r.standard_normal(m + 1)
    sig = -2.0 - 0.6 * np.arange(ns) + 0.5j * (np.arange(ns) % 2)
    beta = np.concatenate([[1.0], r.standard_normal(ns - 1) + 1j * r.standard_normal(ns - 1)])
    D, s, bn, nrm = (torch.zeros(sh, dtype=dt, device="cuda") for sh, dt in (
        ((ns, m), torch.complex128), ((m + 1,), torch.complex128), ((ns,), torch.complex128), ((ns,), torch.float64)))
    g.gdr_dense_gmres_sh(ctx, m, sig, dev(np.ascontiguousarray(H.T)), dev(c), dev(beta), D, s, bn, nrm)
    I = np.eye(m + 1, m)
    d1 = np.linalg.lstsq(H - sig[0] * I, c, rcond=None)[0]
    s1 = c - (H - sig[0] * I) @ d1

    def close(got, ref, cond):
        assert np.linalg.norm(got - ref) <= 1e-13 * cond * max(np.linalg.norm(ref), np.linalg.norm(c) / cond)

    cond = np.linalg.cond(H - sig[0] * I)
    close(D[0].cpu().numpy(), d1, cond)
    close(s.cpu().numpy(), s1, cond)
    for i in range(1, ns):
        M = np.concatenate([H - sig[i] * I, s1[:, None]], 1)
        y = np.linalg.solve(M, beta[i] * c)
        ci = np.linalg.cond(M)
        close(D[i].cpu().numpy(), y[:-1], ci)
        close(bn[i:i + 1].cpu().numpy(), y[-1:], ci)
