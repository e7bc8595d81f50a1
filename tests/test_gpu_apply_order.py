"""gdr_op_apply on Wilson vectors: the reordering at the C interface (runs on a GB300; -m gpu).

The matvec reorders its input in tiles of 64 sites and stores its output site-major from
shared memory, a warp's 32 sites at a time; up to 16 shifts travel by value.  Cases: V a
multiple of neither (ragged tiles and warps), 17 columns (shifts copied), every kernel form,
and complex64 vectors that start 8 bytes off a 16-byte boundary (element-wise reordering).
Against the oracle's operator: FP64 1e-13, complex64 1e-6 of the result's norm (a site sums
~200 products of O(1) terms), as in the other matvec tests."""
import numpy as np
import pytest

import workloads as W
from oracle import WilsonOperator
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_0707_0502_gb300 as g  # noqa: E402

DIMS = [(2, 2, 2, 2), (3, 5, 3, 5), (4, 4, 4, 6), (7, 3, 5, 4)]


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = g.gdr_create(0)
    yield c
    g.gdr_destroy(c)


@pytest.mark.parametrize("dims", DIMS, ids=str)
@pytest.mark.parametrize("prec", [g.GDR_PREC_FP64, g.GDR_PREC_MIXED], ids=["fp64", "c64"])
@pytest.mark.parametrize("form,ncol,offset", [(None, 1, 0), (0, 3, 0), (1, 2, 0), (2, 3, 0), (2, 17, 0), (None, 2, 1)])
def test_apply_orders(ctx, dims, prec, form, ncol, offset):
    f64 = prec == g.GDR_PREC_FP64
    if f64 and (form == 2 or offset):
        pytest.skip("complex64 only")
    links = W.su3_links(dims, 0.4, W.rng(3, 0))
    A = WilsonOperator(dims, links, diag_a=0.3)
    op = g.gdr_op_wilson(ctx, dims, dev(links), 0.3, g.GDR_LINK_C64)
    if form is not None:
        g.gdr_op_set_shape(op, prec, ncol, form, 64 if form == 2 else 128, 1)
    rng = np.random.default_rng(sum(dims) + ncol)
    X = rng.standard_normal((ncol, A.n)) + 1j * rng.standard_normal((ncol, A.n))
    sig = rng.standard_normal(ncol) + 1j * rng.standard_normal(ncol)
    dt = torch.complex128 if f64 else torch.complex64
    buf = [torch.zeros(ncol * A.n + 1, dtype=dt, device="cuda") for _ in range(2)]
    Xd, Yd = (b[offset: offset + ncol * A.n].view(ncol, A.n) for b in buf)
    Xd.copy_(dev(X, dt))
    g.gdr_op_apply(ctx, op, prec, sig, Xd, Yd)
    g.gdr_op_apply(ctx, op, prec, sig, Xd, Xd)      # in place: the input is copied first
    for c in range(ncol):
        x = Xd.new_tensor(X[c]).cpu().numpy().astype(complex)
        ref = A.matvec(x) - sig[c] * x
        for got in (Yd, Xd):
            err = np.linalg.norm(got[c].cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err <= (1e-13 if f64 else 1e-6), (c, err)
    g.gdr_op_destroy(op)
