"""Caller's arrays that start 8 bytes off a 16-byte boundary (runs on a GB300; -m gpu).

The C interface passes c128 arrays as interleaved doubles and asks for no more than a double's
alignment.  Wilson vectors are then reordered word by word: the same permutation, so every
call gives bit by bit what it gives for the same values at an aligned address."""
import ctypes

import numpy as np
import pytest

from tests.gpu_util import dev, small_wilson

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


@pytest.fixture(scope="module")
def wilson(ctx):
    p, A = small_wilson(dims=(3, 3, 5, 3), nshift=2, nrhs=2)
    op = g.make_operator(ctx, p)
    yield p, A, op
    g.gdr_op_destroy(op)


def _real(t):
    return torch.view_as_real(t).reshape(-1)


class _Off:
    """Doubles on the device, the first one 8 bytes behind a 16-byte boundary."""

    def __init__(self, values):
        v = _real(values)
        self.buf = torch.full((v.numel() + 2,), -7.0, dtype=torch.float64, device="cuda")
        assert self.buf.data_ptr() % 16 == 0
        self.buf[1:-1] = v
        self.ptr = self.buf.data_ptr() + 8

    def get(self, like):
        assert self.buf[0] == -7.0 and self.buf[-1] == -7.0        # nothing around the array is written
        return torch.view_as_complex(self.buf[1:-1].clone().view(-1, 2)).view(like.shape)


@pytest.mark.parametrize("prec", [g.GDR_PREC_FP64, g.GDR_PREC_MIXED], ids=["fp64", "mixed"])
def test_wilson_solves(ctx, wilson, prec):
    p, A, op = wilson
    B = dev(p.B.T)
    X = torch.zeros((2, 2, p.n), dtype=torch.complex128, device="cuda")
    prm = g.gdr_params_default(m=p.m, k=p.k, m_proj=p.m_proj, tol=1e-8, prec=prec)
    sig = np.ascontiguousarray(p.sigma, complex)
    st, rep, defl = g.gdr_solve_multishift(ctx, op, sig, B, X, prm, want_defl=True)
    assert st == g.GDR_OK and defl
    Bo, Xo, rp, dh = _Off(B), _Off(torch.zeros_like(X)), g.gdr_report(), ctypes.c_void_p()
    L = g.lib()
    st = L.gdr_solve_multishift(ctx, op, 2, sig.ctypes.data, 2, Bo.ptr, Xo.ptr, ctypes.byref(prm), ctypes.byref(dh),
                                ctypes.byref(rp))
    assert st == g.GDR_OK
    assert torch.equal(Xo.get(X), X)
    Y = torch.zeros_like(X)
    g.gdr_solve_proj(ctx, op, defl, sig, B, Y, prm)
    Yo = _Off(torch.zeros_like(X))
    assert L.gdr_solve_proj(ctx, op, defl, 2, sig.ctypes.data, 2, Bo.ptr, Yo.ptr, ctypes.byref(prm),
                            ctypes.byref(rp)) in (g.GDR_OK, g.GDR_ENOCONV)
    assert torch.equal(Yo.get(Y), Y)
    V = torch.zeros((p.k + 1, p.n), dtype=torch.complex128, device="cuda")
    g.gdr_defl_export(ctx, defl, V)
    Vo = _Off(torch.zeros_like(V))
    assert L.gdr_defl_export(ctx, defl, Vo.ptr, None, None) == g.GDR_OK
    assert torch.equal(Vo.get(V), V)
    for h in (defl, dh):
        g.gdr_defl_destroy(h)


def test_wilson_matvec_and_cycle_fp64(ctx, wilson):
    p, A, op = wilson
    r = np.random.default_rng(1)
    X = dev(r.standard_normal((3, p.n)) + 1j * r.standard_normal((3, p.n)))
    Y = torch.zeros_like(X)
    sig = np.ascontiguousarray([0.0, 0.5j, 1.0], complex)
    g.gdr_op_apply(ctx, op, g.GDR_PREC_FP64, sig, X, Y)
    Xo, Yo = _Off(X), _Off(Y * 0)
    assert g.lib().gdr_op_apply(ctx, op, g.GDR_PREC_FP64, 3, sig.ctypes.data, Xo.ptr, Yo.ptr) == g.GDR_OK
    assert torch.equal(Yo.get(Y), Y)
    m = 6
    V = torch.zeros((m + 1, p.n), dtype=torch.complex128, device="cuda")
    V[0] = X[0] / torch.linalg.vector_norm(X[0])
    H = torch.zeros((m, m + 1), dtype=torch.complex128, device="cuda")
    Vo, Ho, me = _Off(V), _Off(H), ctypes.c_int()
    g.gdr_arnoldi_cycle(ctx, op, g.GDR_PREC_FP64, V, 0, m, H)
    assert g.lib().gdr_arnoldi_cycle(ctx, op, g.GDR_PREC_FP64, Vo.ptr, 0, m, Ho.ptr, 0, ctypes.byref(me)) == g.GDR_OK
    assert torch.equal(Vo.get(V), V) and torch.equal(Ho.get(H), H)


@pytest.mark.parametrize("prec,ncol", [(g.GDR_PREC_MIXED, 12), (g.GDR_PREC_MIXED, 3), (g.GDR_PREC_FP64, 3)])
def test_projection_dots(ctx, prec, ncol):
    """C on the tensor cores (8 columns and more) and on the CUDA cores."""
    n, nv = 300, 9
    r = np.random.default_rng(ncol)
    dt = torch.complex128 if prec == g.GDR_PREC_FP64 else torch.complex64
    V, R = (dev(r.standard_normal((k, n)) + 1j * r.standard_normal((k, n)), dt) for k in (nv, ncol))
    C = torch.zeros((ncol, nv), dtype=torch.complex128, device="cuda")
    g.gdr_basis_dot(ctx, prec, n, nv, V, ncol, R, n, C)
    Co = _Off(torch.zeros_like(C))
    assert g.lib().gdr_basis_dot(ctx, prec, n, nv, V.data_ptr(), ncol, R.data_ptr(), n, Co.ptr, 0) == g.GDR_OK
    assert torch.equal(Co.get(C), C)


@pytest.mark.parametrize("n,nv,ncol,pad,offv,offr", [
    (3001, 21, 1, 0, 0, 0),       # odd n: every second vector of V starts off a boundary
    (3001, 60, 40, 0, 0, 0),      # more vectors than one pass of the element-wise form takes
    (3001, 97, 1, 0, 0, 0),
    (300, 60, 3, 1, 0, 0),        # odd column stride of R
    (300, 60, 2, 0, 1, 0),        # V, R starting 8 bytes off
    (300, 7, 1, 0, 0, 1),
    (300, 60, 12, 0, 1, 1),
    (1, 2, 1, 0, 0, 0),
])
def test_projection_dots_of_unaligned_vectors(ctx, n, nv, ncol, pad, offv, offr):
    """Element by element |dot - exact| <= 2^-16 S, S = sum |v||r| over the real products: a thread
    adds at most 64 complex products in FP32 (three roundings each) before FP64 takes over."""
    r = np.random.default_rng(n + nv)
    V, R = ((r.standard_normal((k, n)) + 1j * r.standard_normal((k, n))).astype(np.complex64) for k in (nv, ncol))
    Vb = torch.zeros(nv * n + 1, dtype=torch.complex64, device="cuda")
    Rb = torch.full(((n + pad) * ncol + 1,), float("nan"), dtype=torch.complex64, device="cuda")
    Vd = Vb[offv: offv + nv * n]
    Rd = Rb[offr: offr + (n + pad) * ncol]
    Vd.copy_(dev(V).view(-1))
    Rd.view(ncol, n + pad)[:, :n] = dev(R)
    C = torch.zeros((ncol, nv), dtype=torch.complex128, device="cuda")
    g.gdr_basis_dot(ctx, g.GDR_PREC_MIXED, n, nv, Vd, ncol, Rd, n + pad, C, g.GDR_FLAG_NO_TENSOR_CORES)
    got = C.cpu().numpy()
    Vx, Rx = V.astype(complex), R.astype(complex)
    exact = Rx @ Vx.conj().T
    S = (np.abs(Rx.real) + np.abs(Rx.imag)) @ (np.abs(Vx.real) + np.abs(Vx.imag)).T
    assert (np.abs(got - exact) <= 2.0 ** -16 * S).all()


def test_unaligned_elements_are_refused(ctx, wilson):
    """Arrays that kernels read element by element: GDR_EINVAL before any work, each in turn."""
    _, _, wop = wilson
    L, n, m, k = g.lib(), 12, 4, 2
    op = g.gdr_op_csr(ctx, dev(np.arange(n + 1, dtype=np.int32)), dev(np.arange(n, dtype=np.int32)),
                      dev(np.ones(n, complex)))
    buf = torch.zeros(4000, dtype=torch.float64, device="cuda")
    sig = np.zeros(8, complex)
    F64, C64 = g.GDR_PREC_FP64, g.GDR_PREC_MIXED
    A = buf.data_ptr()
    # (call with the pointers p[0], p[1], ...; per pointer how far off it may not be, in bytes)
    calls = [
        (lambda p: L.gdr_op_apply(ctx, op, F64, 1, sig.ctypes.data, p[0], p[1]), [8, 8]),
        (lambda p: L.gdr_op_apply(ctx, op, C64, 1, sig.ctypes.data, p[0], p[1]), [4, 4]),
        (lambda p: L.gdr_op_apply(ctx, wop, C64, 1, sig.ctypes.data, p[0], p[1]), [4, 4]),
        (lambda p: L.gdr_arnoldi_step(ctx, op, F64, p[0], 0, A), [8]),
        (lambda p: L.gdr_arnoldi_step(ctx, op, C64, p[0], 0, A), [8]),
        (lambda p: L.gdr_arnoldi_cycle(ctx, wop, C64, p[0], 0, 1, A, 0, None), [4]),
        (lambda p: L.gdr_dense_gmres_sh(ctx, m, 1, A, A, sig.ctypes.data, A, A, p[0], p[1], A), [8, 8]),
        (lambda p: L.gdr_dense_gmres_sh_noalloc(ctx, m, 1, A, A, sig.ctypes.data, A, A, p[0], p[1], A), [8, 8]),
        (lambda p: L.gdr_dense_ls(ctx, F64, m, sig.ctypes.data, p[0], p[1], A, p[2]), [8] * 3),
        (lambda p: L.gdr_dense_restart(ctx, F64, m, k, sig.ctypes.data, *p), [8] * 6),
        (lambda p: L.gdr_basis_update(ctx, F64, n, 2, p[0], p[1], 1, 1, p[2]), [8] * 3),
        (lambda p: L.gdr_basis_update(ctx, C64, n, 2, p[0], p[1], 1, 1, p[2]), [4, 8, 8]),
        (lambda p: L.gdr_basis_dot(ctx, F64, n, 2, p[0], 1, p[1], n, A, 0), [8, 8]),
        (lambda p: L.gdr_basis_dot(ctx, C64, n, 2, p[0], 1, p[1], n, A, 0), [4, 4]),
        (lambda p: L.gdr_basis_residual_update(ctx, F64, n, 2, p[0], 1, p[1], p[2], n, 0), [8] * 3),
        (lambda p: L.gdr_basis_residual_update(ctx, C64, n, 2, p[0], 1, p[1], p[2], n, 0), [4, 8, 4]),
    ]
    for i, (call, offs) in enumerate(calls):
        for q, off in enumerate(offs):
            p = [A] * len(offs)
            p[q] += off
            assert call(p) == g.GDR_EINVAL, (i, q)
    import ctypes as ct
    h, dims = ct.c_void_p(), (ct.c_int * 4)(2, 2, 2, 2)
    assert L.gdr_op_wilson(ctx, dims, 0.0, A + 8, g.GDR_LINK_C64, ct.byref(h)) == g.GDR_EINVAL and not h.value
    torch.cuda.synchronize()
    assert not buf.any()
    g.gdr_op_destroy(op)
