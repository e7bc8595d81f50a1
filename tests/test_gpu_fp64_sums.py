"""FP64 sums of complex products: one rounding per term at the sum's magnitude (runs on a
GB300; -m gpu).

A sum of N products formed one by one rounds at most once per term in each accumulator, so
with all partial sums in [1, 2) each part is off by at most N half-units, N 2^-53 (plus two for
the last additions).  The data make the first term 1 and, in every further one, the product
with the real parts half a unit of the last place and a little (it rounds up) and the other a
quarter unit downwards (it rounds away): accumulators that round twice a term are off by
1.5 (N - 1) 2^-53.  Exact values by rational arithmetic."""
from fractions import Fraction as F

import numpy as np
import pytest

from tests.gpu_util import dev, host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_0707_0502_gb300 as g  # noqa: E402

HALF = 2.0 ** -53                      # half a unit in the last place of [1, 2)
BIG, SMALL = HALF * (1 + 2.0 ** -10), HALF


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    c = g.gdr_create(0)
    yield c
    g.gdr_destroy(c)


def _exact(terms):
    """Real and imaginary part of sum a b over (a, b), exactly."""
    re, im = F(0), F(0)
    for a, b in terms:
        ax, ay, bx, by = F(a.real), F(a.imag), F(b.real), F(b.imag)
        re += ax * bx - ay * by
        im += ax * by + ay * bx
    return re, im


def _check(got, exact, n):
    for x, e in zip((got.real, got.imag), exact):
        assert abs(F(float(x)) - e) <= (n + 2) * F(HALF), float(abs(F(float(x)) - e) / F(HALF))


@pytest.mark.parametrize("nv,nout,nx", [(40, 2, 1), (40, 1, 0), (81, 30, 2), (40, 0, 1), (40, 0, 3), (97, 0, 12),
                                        (97, 0, 30)])
def test_basis_update(ctx, nv, nout, nx):
    n = 70
    V = np.full((nv, n), BIG + 1j * SMALL, complex)
    V[0] = 1
    C = np.full((nout + nx, nv), 1 + 0.5j, complex)
    C[:, 0] = 1
    Vd, X = dev(V), torch.zeros((max(nx, 1), n), dtype=torch.complex128, device="cuda")
    g.gdr_basis_update(ctx, g.GDR_PREC_FP64, n, nv, Vd, dev(C), nout, nx, X)
    exact = _exact(zip(V[:, 0], C[0]))
    out = np.concatenate([host(Vd)[:nout], host(X)[:nx]])
    assert (out == out[0, 0]).all()
    _check(out[0, 0], exact, nv)


@pytest.mark.parametrize("nv,ncol", [(40, 2), (40, 5), (97, 3)])
def test_residual_update(ctx, nv, ncol):
    n = 70
    V = np.full((nv, n), BIG + 1j * SMALL, complex)
    V[0] = 1
    T = np.full((ncol, nv), 1 + 0.5j, complex)
    T[:, 0] = 1
    R = torch.zeros((ncol, n), dtype=torch.complex128, device="cuda")
    g.gdr_basis_residual_update(ctx, g.GDR_PREC_FP64, n, nv, dev(V), ncol, dev(T), R, n)
    assert (R == R[0, 0]).all()
    _check(host(R)[0, 0], _exact(zip(V[:, 0], T[0])), nv)


@pytest.mark.parametrize("nv,ncol", [(2, 2), (30, 3)])
def test_shared_basis_dot(ctx, nv, ncol):
    """A thread's sum runs over every 32nd row of a 128-row tile and over up to 16 tiles that lie
    as many tiles apart as there are blocks (two per SM): one thread's 64 terms, the rest zero."""
    S = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    n = 16 * S * 128
    rows = (128 * S * np.arange(16)[:, None] + 32 * np.arange(4)[None, :]).ravel()
    v = np.full(64, BIG - 1j * SMALL, complex)  # conj(v) enters
    v[0] = 1
    w = np.full(64, 1 + 0.5j, complex)
    w[0] = 1
    V = torch.zeros((nv, n), dtype=torch.complex128, device="cuda")
    R = torch.zeros((ncol, n), dtype=torch.complex128, device="cuda")
    V[:, dev(rows)] = dev(v)
    R[:, dev(rows)] = dev(w)
    C = torch.zeros((ncol, nv), dtype=torch.complex128, device="cuda")
    g.gdr_basis_dot(ctx, g.GDR_PREC_FP64, n, nv, V, ncol, R, n, C)
    assert (C == C[0, 0]).all()
    _check(host(C)[0, 0], _exact(zip(v.conj(), w)), 64)


def _reduced(ctx, H, c):
    m = H.shape[1]
    z = lambda *sh: torch.zeros(sh, dtype=torch.complex128, device="cuda")
    D, s, bn = z(1, m), z(m + 1), z(1)
    g.gdr_dense_gmres_sh(ctx, m, [0.0], dev(np.ascontiguousarray(H.T)), dev(c), dev(np.ones(1, complex)), D, s, bn,
                         torch.zeros(1, dtype=torch.float64, device="cuda"))
    return host(D)[0], host(s)


def test_back_substitution(ctx):
    """A unit upper triangle whose first row alone has entries beside the diagonal: nothing to
    reflect, y_j = c_j below, y_0 = c_0 - sum h_0j y_j."""
    m = 40
    H = np.eye(m + 1, m, dtype=complex)
    H[0, 1:] = -BIG - 0.5j * SMALL
    c = np.full(m + 1, 1 + 1j)
    y, _ = _reduced(ctx, H, c)
    assert (y[1:] == 1 + 1j).all()
    _check(y[0], _exact([(c[0], 1 + 0j)] + [(-H[0, j], y[j]) for j in range(1, m)]), m)


def test_least_squares_residual(ctx):
    """s = c - H y in its last component, for the y that the call returns."""
    m = 40
    H = np.eye(m + 1, m, dtype=complex)
    H[m] = -BIG - 0.5j * SMALL
    c = np.full(m + 1, 1 + 1j)
    y, s = _reduced(ctx, H, c)
    assert np.abs(y - (1 + 1j)).max() < 1e-14
    _check(s[m], _exact([(c[m], 1 + 0j)] + [(-H[m, j], y[j]) for j in range(m)]), m + 1)


@pytest.mark.parametrize("ns", [2, 9])
def test_reflected_right_hand_side(ctx, ns):
    """beta_new of a shift at which H is a unit matrix over a small last row t: m reflectors each take
    t_j c_j from the last component of c, and beta_new (s_m - sum t_j s_j) = c_m - sum t_j c_j.
    The base shift lies far away, so that s differs from c in the last component only.  (Two
    shifts: one cluster; nine: two launches.)"""
    m = 80
    H = np.eye(m + 1, m, dtype=complex)
    H[m] = -BIG - 0.5j * SMALL
    c = np.full(m + 1, 1 + 1j)
    c[m] = 1
    z = lambda *sh: torch.zeros(sh, dtype=torch.complex128, device="cuda")
    D, s, bn = z(ns, m), z(m + 1), z(ns)
    g.gdr_dense_gmres_sh(ctx, m, [-1023.0] + [0.0] * (ns - 1), dev(np.ascontiguousarray(H.T)), dev(c),
                         dev(np.ones(ns, complex)), D, s, bn, torch.zeros(ns, dtype=torch.float64, device="cuda"))
    s, bn = host(s), host(bn)
    assert abs(s[m] - 1) < 1e-14 and np.abs(s[:m]).max() < 1e-12
    num = _exact([(c[m], 1 + 0j)] + [(-H[m, j], c[j]) for j in range(m)])
    den = _exact([(s[m], 1 + 0j)] + [(-H[m, j], s[j]) for j in range(m)])
    d2 = den[0] ** 2 + den[1] ** 2
    want = (num[0] * den[0] + num[1] * den[1]) / d2, (num[1] * den[0] - num[0] * den[1]) / d2
    for b in bn[1:]:
        _check(b, want, m + 10)   # ten more roundings for the quotient
