"""The projection of vectors longer than 32-bit TMA coordinates reach (runs on a GB300; -m gpu).

2^30 + 64 complex64 entries are 2^31 + 128 floats.  All but a few entries on both sides of that
line are zero, and those are small integers, so dots and updates are exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_0707_0502_gb300 as g  # noqa: E402

N, NCOL = (1 << 30) + 64, 8


def test_entries_behind_the_32_bit_line():
    if torch.cuda.mem_get_info()[0] < 120 << 30:
        pytest.skip("needs 90 GB of device memory")
    import __graft_entry__
    __graft_entry__.build()
    ctx = g.gdr_create(0)
    rows = torch.tensor([0, 1, 63, 64, (1 << 29) + 5, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, N - 1], device="cuda")
    r = np.random.default_rng(0)
    v = (r.integers(-4, 5, 9) + 1j * r.integers(-4, 5, 9)).astype(np.complex64)
    w = (r.integers(-4, 5, (NCOL, 9)) + 1j * r.integers(-4, 5, (NCOL, 9))).astype(np.complex64)
    t = r.integers(-4, 5, (NCOL, 1)) + 1j * r.integers(-4, 5, (NCOL, 1))
    V = torch.zeros((1, N), dtype=torch.complex64, device="cuda")
    R = torch.zeros((NCOL, N), dtype=torch.complex64, device="cuda")
    V[:, rows] = torch.as_tensor(v, device="cuda")
    R[:, rows] = torch.as_tensor(w, device="cuda")
    C = torch.zeros((NCOL, 1), dtype=torch.complex128, device="cuda")
    g.gdr_basis_dot(ctx, g.GDR_PREC_MIXED, N, 1, V, NCOL, R, N, C)
    assert np.array_equal(C.cpu().numpy()[:, 0], w.astype(complex) @ v.conj().astype(complex))
    g.gdr_basis_residual_update(ctx, g.GDR_PREC_MIXED, N, 1, V, NCOL, torch.as_tensor(t, device="cuda"), R, N)
    assert np.array_equal(R[:, rows].cpu().numpy(), (w + t * v).astype(np.complex64))
    assert int(sum((R[c] != 0).sum() for c in range(NCOL))) == int(np.count_nonzero(w + t * v))
    g.gdr_destroy(ctx)
    del V, R
    torch.cuda.empty_cache()
