"""Steps of the complex128 bond SVD on their own (gpeps_selftest_core)."""
import ctypes
import math

import numpy as np
import pytest
import torch

from ._gpu_util import gpu_lib

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps


def _run(which, a, b):
    gpu_lib()
    from paper_2309_15642_gb300 import _abi
    x, y = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (a, b))
    out = torch.empty_like(x)
    assert _abi.load().gpeps_selftest_core(which, len(a), x.data_ptr(), y.data_ptr(), out.data_ptr(),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _two_products(x, y):
    """x y as a sum of two doubles (Dekker, with Veltkamp's splitting)."""
    def split(v):
        t = 134217729.0 * v
        hi = t - (t - v)
        return hi, v - hi
    p, (xh, xl), (yh, yl) = x * y, split(x), split(y)
    return p, ((xh * yh - p) + xh * yl + xl * yh) + xl * yl


@pytest.mark.parametrize("n", [48, 64, 128, 256])
def test_digit_product_is_no_less_accurate_than_fp64(n):
    """Gaussian rows: every real output against its exact value, in units of 2^-53 of the two rows'
    powers of two.  They have to be no worse than FP64 products summed in order, and unbiased
    within five standard errors."""
    rng = np.random.default_rng(n)
    a, b = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)) for _ in range(2))
    got = _run(0, a, b)
    rows = rng.permutation(n)[:16]
    unit = [2.0 ** np.frexp(np.maximum(np.abs(v.real), np.abs(v.imag)).max(1))[1] for v in (a, b)]
    err, plain = [], []
    for i in rows:
        # re: (ar, ai) . (br, bi), im: (ar, -ai) . (bi, br)
        for part, x, y in ((got[i].real, np.r_[a[i].real, a[i].imag], np.c_[b.real, b.imag]),
                           (got[i].imag, np.r_[a[i].real, -a[i].imag], np.c_[b.imag, b.real])):
            p, q = _two_products(x[None, :], y)
            scale = unit[0][i] * unit[1] * 2.0 ** -53
            exact = [math.fsum(np.r_[u, v]) for u, v in zip(p, q)]
            rest = [math.fsum(np.r_[u, v, -w]) for u, v, w in zip(p, q, exact)]
            err.append(((part - exact) - rest) / scale)
            s = np.zeros(n)
            for k in range(x.size):
                s = s + p[:, k]
            plain.append(((s - exact) - rest) / scale)
    err, plain = np.array(err), np.array(plain)
    rms, ref = np.sqrt((err ** 2).mean()), np.sqrt((plain ** 2).mean())
    assert rms <= ref
    assert abs(err.mean()) <= 5 * rms / np.sqrt(err.size)


@pytest.mark.parametrize("angle", [1e-7, 1.9e-5])
@pytest.mark.parametrize("n", [48, 64, 128, 256])
def test_correction_is_unitary(n, angle):
    """Columns of norms 2 to 1 turned away from orthogonality by exp(X), all angles of one size and
    sign (the largest |X| they allow).  A correction multiplies them by a unitary factor, up to
    sqrt(n) 2^-53 an element each from X^4 and from the rounding of X^2, 2 eps from the digit
    products and about 2 sqrt(n) eps from the solve that recovers the factor here: held to
    4 sqrt(n) eps, the singular values too.  A factor as unitary as its angles are small is
    1e-14, 5e-14 and 2e-13 off at 64, 128 and 256 columns.  At 1e-7, where the pass is meant to work,
    the largest overlap falls a hundredfold."""
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    w, v = np.linalg.eigh(1j * angle * (np.triu(np.ones((n, n)), 1) - np.tril(np.ones((n, n)), -1)))
    z = (q * np.linspace(2.0, 1.0, n)) @ ((v * np.exp(1j * w)) @ v.conj().T)
    out = _run(1, np.ascontiguousarray(z.T), np.zeros((3 * n, n + 1), np.complex128)).T
    u = np.linalg.solve(z, out)
    assert np.abs(u.conj().T @ u - np.eye(n)).max() <= 4 * np.sqrt(n) * EPS
    before, after = (np.linalg.svd(m, compute_uv=False) for m in (z, out))
    assert np.abs(before - after).max() <= 2.0 * 4 * np.sqrt(n) * EPS
    if angle == 1e-7:
        def far(m):
            m = m / np.linalg.norm(m, axis=0)
            return np.abs(m.conj().T @ m - np.eye(n)).max()
        assert far(out) <= far(z) / 100


def test_rejects_bad_arguments():
    gpu_lib()
    from paper_2309_15642_gb300 import _abi
    lib = _abi.load()
    x = torch.zeros(64, dtype=torch.float64, device="cuda").data_ptr()
    for which, n, p in ((7, 4, x), (0, 3, x), (0, 0, x), (0, 258, x), (0, 4, None)):
        assert lib.gpeps_selftest_core(which, n, p, p, p, None) == _abi.GPEPS_EINVAL
