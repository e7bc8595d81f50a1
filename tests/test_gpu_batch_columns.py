"""gdr_op_apply on a CSR batch: one column per problem at most (runs on a GB300; -m gpu)."""
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


def test_batch_matvec_beyond_its_problems_is_refused(ctx):
    rp, cl, vl = np.arange(5, dtype=np.int32), np.arange(4, dtype=np.int32), np.ones(4, complex)
    op = g.gdr_op_csr_batch(ctx, [4, 4], [4, 4], dev(np.tile(rp, 2)), dev(np.tile(cl, 2)), dev(np.tile(vl, 2)))
    X = torch.ones((3, 4), dtype=torch.complex128, device="cuda")
    Y = torch.zeros_like(X)
    with pytest.raises(g.GdrError) as e:
        g.gdr_op_apply(ctx, op, g.GDR_PREC_FP64, [0, 0, 0], X, Y)
    assert e.value.status == g.GDR_EINVAL
    for ncol in (1, 2):  # fewer columns than problems: the first problems
        Y.zero_()
        g.gdr_op_apply(ctx, op, g.GDR_PREC_FP64, [0.5] * ncol, X[:ncol].contiguous(), Y[:ncol])
        assert (Y[:ncol] == 0.5).all() and not Y[ncol:].any()
    g.gdr_op_destroy(op)
