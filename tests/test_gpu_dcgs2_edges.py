"""DCGS2 Arnoldi cycles at the edges of the dot pass's tiling (runs on a GB300; -m gpu).

A warp's slab is 32 x (2 to 8) units of two complex64 elements, a block takes eight, and short
vectors split their basis over several blocks: vectors shorter than one slab, one element pair
on either side of slab and block boundaries, one step, and as many steps as the largest basis
allows.  Checked, as the other complex64 cycles, by what defines them: orthonormal to 1e-5 and
the Arnoldi relation to 1e-5 of ||Hbar|| (complex64 rounding, u = 6e-8, of up to 1e3 terms)."""
import numpy as np
import pytest

from tests.gpu_util import dev, host

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


@pytest.mark.parametrize("n,m", [(8, 3), (126, 20), (128, 1), (130, 20), (510, 33), (514, 96), (4094, 40), (4098, 40),
                                 (16386, 25), (70002, 31)])
def test_cycle_sizes(ctx, n, m):
    r = np.random.default_rng(n)
    # a periodic three-point operator with random complex coefficients
    col = np.stack([(np.arange(n) + o) % n for o in (-1, 0, 1)], 1).astype(np.int32)
    val = r.standard_normal((n, 3)) + 1j * r.standard_normal((n, 3))
    op = g.gdr_op_csr(ctx, dev(np.arange(0, 3 * n + 1, 3, dtype=np.int32)), dev(col.ravel()), dev(val.ravel()))
    V = torch.zeros((m + 1, n), dtype=torch.complex64, device="cuda")
    v0 = r.standard_normal(n) + 1j * r.standard_normal(n)
    V[0] = dev(v0 / np.linalg.norm(v0), torch.complex64)
    H = torch.zeros((m, m + 1), dtype=torch.complex128, device="cuda")
    assert g.gdr_arnoldi_cycle(ctx, op, g.GDR_PREC_MIXED, V, 0, m, H) == m
    Q, Hb = host(V).T.astype(complex), host(H).T
    assert np.abs(Q.conj().T @ Q - np.eye(m + 1)).max() <= 1e-5
    AQ = np.einsum("nk,nkj->nj", val.astype(np.complex64).astype(complex), Q[col][:, :, :m])
    assert np.linalg.norm(AQ - Q @ Hb) <= 1e-5 * np.linalg.norm(Hb)
    g.gdr_op_destroy(op)
