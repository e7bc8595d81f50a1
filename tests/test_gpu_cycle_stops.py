"""gdr_arnoldi_cycle that meets a non-finite vector (runs on a GB300; -m gpu).

A e_i = e_{i+1}, except A e_2 = 1e25 e_3, whose squared norm overflows complex64: from e_0 the
cycle forms e_0 and e_1 and stops at step 2 with GDR_ENAN, before v_2 exists.  The columns it
has not formed are zero, whatever the library's workspace holds of an earlier cycle."""
import numpy as np
import pytest

from tests.gpu_util import dev, host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_0707_0502_gb300 as g  # noqa: E402


@pytest.mark.parametrize("flags", [0, g.GDR_FLAG_CGS2], ids=["dcgs2", "cgs2"])
def test_columns_not_formed_are_zero(flags):
    import __graft_entry__
    __graft_entry__.build()
    ctx = g.gdr_create(0)
    n, m = 16, 8
    r = np.random.default_rng(0)
    rowptr = dev(np.arange(n + 1, dtype=np.int32))
    col = dev(np.arange(n, dtype=np.int32) - 1 + n * (np.arange(n) == 0).astype(np.int32))
    val = np.ones(n, complex)
    plain = g.gdr_op_csr(ctx, rowptr, col, dev(val + r.standard_normal(n)))
    val[3] = 1e25
    op = g.gdr_op_csr(ctx, rowptr, col, dev(val))
    H = torch.zeros((m, m + 1), dtype=torch.complex128, device="cuda")
    V = torch.zeros((m + 1, n), dtype=torch.complex64, device="cuda")
    v = r.standard_normal(n)
    V[0] = dev(v / np.linalg.norm(v), torch.complex64)
    g.gdr_arnoldi_cycle(ctx, plain, g.GDR_PREC_MIXED, V, 0, m, H, flags)
    assert np.all(np.abs(host(V)).sum(1) > 0)  # a full basis, in the workspace too
    V.fill_(3.0)
    V[0] = 0
    V[0, 0] = 1
    with pytest.raises(g.GdrError) as e:
        g.gdr_arnoldi_cycle(ctx, op, g.GDR_PREC_MIXED, V, 0, m, H, flags)
    assert e.value.status == g.GDR_ENAN
    got = host(V)
    assert np.array_equal(got[:2], np.eye(2, n))
    if not flags:
        assert not got[2:].any()
    else:  # here v_2 = e_2 has been normalised before A v_2 overflows
        assert np.array_equal(got[2], np.eye(3, n)[2]) and not got[4:].any()
    g.gdr_op_destroy(op)
    g.gdr_op_destroy(plain)
    g.gdr_destroy(ctx)
