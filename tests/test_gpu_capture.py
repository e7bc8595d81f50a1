"""gdr_op_apply under stream capture (runs on a GB300; -m gpu).

The shifts are host memory, and a captured call reads them again at each replay: a program
that changes them in place between replays gets the new ones.  Bit by bit what the direct call
gives for the same shifts; up to 16 of them (which a direct call passes by value), 17, and
complex64 vectors 8 bytes off a 16-byte boundary (reordered element by element)."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_0707_0502_gb300 as g  # noqa: E402


@pytest.mark.parametrize("ncol,offset", [(1, 0), (3, 0), (17, 0), (2, 1)])
def test_shifts_at_replay(ncol, offset):
    import __graft_entry__
    __graft_entry__.build()
    s = torch.cuda.Stream()
    ctx = g.gdr_create(0, s)
    dims = (4, 3, 2, 5)
    n = 12 * int(np.prod(dims))
    op = g.gdr_op_wilson(ctx, dims, dev(W.su3_links(dims, 0.4, W.rng(3, 0))), 0.3, g.GDR_LINK_C64)
    r = np.random.default_rng(ncol)
    buf = [torch.zeros(ncol * n + 1, dtype=torch.complex64, device="cuda") for _ in range(2)]
    X, Y = (b[offset: offset + ncol * n].view(ncol, n) for b in buf)
    X.copy_(dev(r.standard_normal((ncol, n)) + 1j * r.standard_normal((ncol, n)), torch.complex64))
    shifts = [r.standard_normal(ncol) + 1j * r.standard_normal(ncol) for _ in range(3)]
    sig = torch.zeros(ncol, dtype=torch.complex128).pin_memory()

    def apply():
        assert g.lib().gdr_op_apply(ctx, op, g.GDR_PREC_MIXED, ncol, sig.data_ptr(), X.data_ptr(),
                                    Y.data_ptr()) == g.GDR_OK

    torch.cuda.synchronize()
    want = []
    for v in shifts:
        sig.copy_(torch.as_tensor(v))
        apply()
        torch.cuda.synchronize()
        want.append(Y.clone())
    assert not torch.equal(want[0], want[1])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
        apply()
    for v, w in list(zip(shifts, want))[::-1]:
        sig.copy_(torch.as_tensor(v))
        Y.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(Y, w)
    del graph
    g.gdr_op_destroy(op)
    g.gdr_destroy(ctx)
