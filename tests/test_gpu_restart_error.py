"""The complex64 restart's error against 64 bits is no larger than FP32's (runs on a GB300; -m gpu).

Whatever form gdr_basis_update chooses, its rms error over orthonormal coefficients is held to
that of the plain FP32 sum (products rounded, one accumulator), which is emulated here with
FMAs in 64 bits.  Both are means over some 10^6 errors of single elements, good to about
0.2%: 2% is allowed.  Basis sizes on both sides of the line between the forms."""
import numpy as np
import pytest

from tests.gpu_util import dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no GPU", allow_module_level=True)

import paper_0707_0502_gb300 as g  # noqa: E402


def _fma32(a, b, c):
    return (a.astype(np.float64) * b + c).astype(np.float32)  # the product of two FP32 values is exact


@pytest.mark.parametrize("nv,nout", [(26, 26), (33, 30), (41, 28), (53, 30), (54, 30), (61, 31), (81, 41), (97, 20)])
def test_error_is_no_larger_than_fp32(nv, nout):
    import __graft_entry__
    __graft_entry__.build()
    ctx = g.gdr_create(0)
    n = 20000
    r = np.random.default_rng(nv)
    V = ((r.standard_normal((nv, n)) + 1j * r.standard_normal((nv, n))) / np.sqrt(2 * n)).astype(np.complex64)
    C = np.linalg.qr(r.standard_normal((nv, nout)) + 1j * r.standard_normal((nv, nout)))[0].T.copy()
    Vd = dev(V)
    g.gdr_basis_update(ctx, g.GDR_PREC_MIXED, n, nv, Vd, dev(C), nout, 0, None)
    exact = C @ V.astype(complex)
    err = np.abs(Vd[:nout].cpu().numpy() - exact)
    c = C.astype(np.complex64)
    re, im = np.zeros((nout, n), np.float32), np.zeros((nout, n), np.float32)
    for i in range(nv):
        a, b, x, y = V[i].real[None], V[i].imag[None], c[:, i].real[:, None], c[:, i].imag[:, None]
        re += _fma32(a, x, -(b * y).astype(np.float64))
        im += _fma32(a, y, (b * x).astype(np.float64))
    plain = np.abs(re + 1j * im.astype(complex) - exact)
    ratio = np.sqrt(np.mean(err ** 2) / np.mean(plain ** 2))
    assert ratio <= 1.02, ratio
    g.gdr_destroy(ctx)
