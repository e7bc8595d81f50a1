"""The restart's basis update on the tensor cores (runs on a GB300; -m gpu).

gdr_basis_update with complex64 vectors forms V[:, 0:nout] <- V C in place and
X[:, i] += V D[:, i] (FP64) by split-TF32 products (three per pair of values).  Element by
element, against numpy's FP64 product of the same complex64 inputs,

    |out - exact| <= 2^-16 S (+ 2^-50 |X|),

S = sum_k |A_mk| |B_kc| over the real form: K = 2 nv <= 194 terms, whose worst-case FP32
accumulation (194 x 2^-24) stays below 2^-16, as do the coefficients' rounding to FP32
(2^-24), the dropped lo*lo product and the low parts' rounding (2^-21 together).  The
median error is held to FP32's level, far from a single TF32 product's 2^-11.

Sizes: row tiles of 64 (ragged ends, fewer rows than one tile), K atoms of 16 vectors (two,
three, six, seven), MMA widths in steps of 16, odd n, and both sides of the lines to the CUDA
cores: fewer than 26 outputs (16 with more than 60 vectors) and coefficients that do not fit
(the CUDA-core form's bound is the same)."""
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


@pytest.mark.parametrize("n,nv,nout,nx", [
    (40, 2, 1, 0),           # few outputs: CUDA cores
    (64, 16, 16, 1),
    (3001, 17, 9, 3),
    (40, 26, 26, 0),         # less than one row tile, the fewest outputs
    (64, 32, 32, 1),         # exactly one tile, two full K atoms, N = 33
    (3001, 33, 23, 3),       # odd n, three K atoms
    (3001, 60, 25, 0),       # the last on the CUDA cores
    (3001, 61, 15, 0),       # the same with more vectors
    (3001, 61, 12, 4),       # N = 16
    (19456, 41, 21, 10),     # two tiles per CTA
    (4097, 81, 41, 0),       # six K atoms
    (100000, 61, 31, 8),     # many tiles per CTA: the ring of K atoms wraps
    (5000, 97, 49, 10),      # the largest basis: seven K atoms
    (2000, 96, 90, 12),      # coefficients beyond shared memory: CUDA cores
])
def test_restart(ctx, n, nv, nout, nx):
    rng = np.random.default_rng(n + nv)
    V = (rng.standard_normal((nv, n)) + 1j * rng.standard_normal((nv, n))).astype(np.complex64)
    V /= np.linalg.norm(V, axis=1, keepdims=True)
    C = rng.standard_normal((nout + nx, nv)) + 1j * rng.standard_normal((nout + nx, nv))
    C *= np.exp(rng.uniform(-3, 3, size=(nout + nx, 1)))
    X = rng.standard_normal((max(nx, 1), n)) + 1j * rng.standard_normal((max(nx, 1), n))
    Vd, Xd = dev(V), dev(X)
    g.gdr_basis_update(ctx, g.GDR_PREC_MIXED, n, nv, Vd, dev(C), nout, nx, Xd)
    V2, X2 = Vd.cpu().numpy(), Xd.cpu().numpy()
    Vx = V.astype(np.complex128)
    P = C @ Vx
    aV = np.abs(Vx.real), np.abs(Vx.imag)
    Sre = np.abs(C.real) @ aV[0] + np.abs(C.imag) @ aV[1]
    Sim = np.abs(C.real) @ aV[1] + np.abs(C.imag) @ aV[0]
    exact = np.concatenate([P[:nout], X[:nx] + P[nout:]])
    got = np.concatenate([V2[:nout].astype(np.complex128), X2[:nx]])
    base = np.concatenate([np.zeros((nout, n)), np.abs(X[:nx])])
    e = np.abs(got.real - exact.real), np.abs(got.imag - exact.imag)
    assert np.all(e[0] <= 2.0 ** -16 * Sre + 2.0 ** -50 * base)
    assert np.all(e[1] <= 2.0 ** -16 * Sim + 2.0 ** -50 * base)
    assert np.median(e[0] / Sre) < 2.0 ** -21
    assert np.array_equal(V2[nout:], V[nout:])       # the other vectors are untouched
    assert np.array_equal(X2[nx:], X[nx:])
